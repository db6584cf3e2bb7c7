"""The U-Net backward's reductions over voxels (weight and bias gradients) at the edges of
their tiles: odd planes, single-voxel levels, rows longer than a run, one and several samples."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import torch.nn.functional as F  # noqa: E402
pytestmark = pytest.mark.gpu

from oracle import unet_oracle as U  # noqa: E402
from paper_2406_13651_gb300 import inputs as I  # noqa: E402


@pytest.fixture(scope="module")
def C():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_13651_gb300 import build, clamp
    build.build()
    clamp.load()
    return clamp


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def _layers(ch):
    off = 0
    for kind, ci, co in U.layer_specs(*ch):
        nw = co * ci * (27 if kind == "conv3" else 8 if kind == "tconv" else 1)
        yield kind, slice(off, off + nw), slice(off + nw, off + nw + co)
        off += nw + co


def _grads(C, ch, p, x, t, dtype, tc=True):
    net = C.UNet(*ch, params=p, dtype=dtype)
    net.set_tensor_cores(tc)
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    net.backward(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), loss)
    net.check()
    return net.get("grads")


def _pre_activations(p, x, ch):
    """Every ReLU layer's pre-activations in FP64."""
    L, out = U.unpack(p.astype(np.float64), ch), []
    h = torch.as_tensor(x.astype(np.float64))[:, None]

    def conv(i, v):
        out.append(F.conv3d(v, L[i][1], L[i][2], padding=1))
        return F.relu(out[-1])

    def up(i, v):
        return F.conv_transpose3d(v, L[i][1], L[i][2], stride=2)

    s1 = conv(1, conv(0, h))
    s2 = conv(3, conv(2, F.max_pool3d(s1, 2)))
    d2 = conv(8, conv(7, torch.cat([up(6, conv(5, conv(4, F.max_pool3d(s2, 2)))), s2], dim=1)))
    conv(11, conv(10, torch.cat([up(9, d2), s1], dim=1)))
    return out


def _problem(ch, shape, B, seed):
    """Parameters, inputs and targets of the first seed whose pre-activations all stay clear of
    zero: one within the FP32 forward error (5e-7 of the layer's mean) may take the other side
    of its ReLU, which changes gradients by a whole voxel's share, whatever sums them."""
    for seed in range(seed, seed + 200):
        p = I.unet_params(ch, seed=seed)
        p[-1] = 0.5
        rng = np.random.default_rng(seed)
        x = rng.uniform(0.0, 2.0, size=(B,) + shape).astype(np.float32)
        t = rng.uniform(0.0, 1.5, size=(B,) + shape).astype(np.float32)
        if all(float(a.abs().min()) > 2e-6 * float(a.abs().mean()) for a in _pre_activations(p, x, ch)):
            return p, x, t
    raise AssertionError("no seed keeps clear of zero")


# FP32 network against exact gradients: 1e-4 as for the other FP32 gradient tests (FP32
# forward and backward through twelve layers)
# (the last two: transposed convs with more channels than one block of their kernels holds)
@pytest.mark.parametrize("shape,B,ch", [((4, 4, 4), 3, (4, 8, 16)), ((12, 4, 20), 2, (4, 8, 16)),
                                        ((4, 8, 136), 1, (4, 8, 16)), ((8, 36, 28), 5, (4, 8, 16)),
                                        ((4, 4, 256), 1, (4, 8, 16)), ((4, 8, 512), 1, (4, 8, 16)),
                                        ((4, 4, 8), 2, (132, 4, 4)), ((8, 4, 4), 1, (4, 20, 36))])
def test_fp32_gradients_match_oracle(C, shape, B, ch):
    p, x, t = _problem(ch, shape, B, 41)
    g = _grads(C, ch, p, x, t, "fp32")
    _, gref = U.loss_and_grad(p.astype(np.float64), x.astype(np.float64), t.astype(np.float64), ch)
    for i, (kind, ws, bs) in enumerate(_layers(ch)):
        assert rel(g[ws], gref[ws]) < 1e-4, (i, kind, "weights")
        assert rel(g[bs], gref[bs]) < 1e-4, (i, kind, "biases")


# BF16 network whose 3x3x3 convs all run on the CUDA cores (no level is a width the tensor
# convs take), so that both settings see the same activations and output gradients and only
# the weight gradients' sums differ: FP32 chains and truncated 16-step tensor chains (3e-7 of
# a same-signed sum) against each other.  1e-5 leaves 30x for cancellation within a layer.
# Widths: below, at and above the 8, 16 and 32 voxel tiles, aligned and not; heights around
# the rows of a tile.
@pytest.mark.parametrize("shape,B,ch", [((4, 4, 4), 3, (4, 8, 16)), ((8, 12, 16), 2, (4, 8, 16)),
                                        ((4, 20, 24), 3, (8, 16, 32)), ((12, 36, 20), 2, (16, 32, 64)),
                                        ((8, 4, 40), 1, (16, 24, 40)), ((4, 68, 72), 2, (12, 20, 64))])
def test_weight_gradients_tensor_cores_match_cuda_cores(C, shape, B, ch):
    p, x, t = _problem(ch, shape, B, 61)
    tc, cc = _grads(C, ch, p, x, t, "bf16", True), _grads(C, ch, p, x, t, "bf16", False)
    for i, (kind, ws, bs) in enumerate(_layers(ch)):
        assert np.isfinite(tc[ws]).all() and np.isfinite(tc[bs]).all()
        assert rel(tc[ws], cc[ws]) < 1e-5, (i, kind, "weights", rel(tc[ws], cc[ws]))
        assert rel(tc[bs], cc[bs]) < 1e-5, (i, kind, "biases", rel(tc[bs], cc[bs]))

