"""The U-Net's bias, 1x1 and transposed-conv gradients, and the 3x3x3 weight gradients formed on the
tensor cores, repeat bit for bit: their partial sums are added in a fixed order."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
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


# many CTAs per sum; an odd coarsest level whose planes are no whole 16-byte groups, ragged channels
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("shape,B,ch", [((32, 32, 32), 6, (16, 32, 64)), ((4, 12, 20), 7, (5, 20, 36))])
def test_gradients_repeat(C, dtype, shape, B, ch):
    net = C.UNet(*ch, params=I.unet_params(ch, seed=3), dtype=dtype)
    rng = np.random.default_rng(8)
    x = torch.from_numpy(rng.uniform(0.0, 2.0, (B,) + shape).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.uniform(0.0, 1.5, (B,) + shape).astype(np.float32)).cuda()
    runs = []
    for _ in range(4):
        net.backward(x, t, torch.zeros((), dtype=torch.float64, device="cuda"))
        runs.append(net.get("grads"))
    net.check()
    off = 0
    for kind, ci, co in U.layer_specs(*ch):
        nw = co * ci * (27 if kind == "conv3" else 8 if kind == "tconv" else 1)
        parts = [slice(off + nw, off + nw + co)] + ([slice(off, off + nw)] if kind != "conv3" else [])
        for s in parts:
            assert np.abs(runs[0][s]).max() > 0
            for r in runs[1:]:
                assert np.array_equal(r[s], runs[0][s]), (kind, ci, co)
        off += nw + co


def test_tensor_core_weight_gradients_repeat(C):
    ch, B, shape = (16, 32, 64), 6, (32, 32, 32)      # chains of 1 k to 10 k terms: all on the tensor cores
    net = C.UNet(*ch, params=I.unet_params(ch, seed=3), dtype="bf16")
    rng = np.random.default_rng(9)
    x = torch.from_numpy(rng.uniform(0.0, 2.0, (B,) + shape).astype(np.float32)).cuda()
    runs = []
    for _ in range(3):
        net.backward(x, 0.5 * x, torch.zeros((), dtype=torch.float64, device="cuda"))
        runs.append(net.get("grads"))
    net.check()
    assert np.array_equal(runs[1], runs[0]) and np.array_equal(runs[2], runs[0])
