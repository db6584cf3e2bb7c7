"""The 3x3x3 weight gradients of BF16 networks against FP64 sums of the same rounded operands.

The networks are made so that one layer's operands are known without rounding: its inputs are
shifted copies of the image (or of its max-pooled half), its output gradient a few exact values.
Sizes lie on both sides of the chain lengths that choose between the tensor cores and the CUDA cores."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import torch.nn.functional as F  # noqa: E402
pytestmark = pytest.mark.gpu

from oracle import unet_oracle as U  # noqa: E402


@pytest.fixture(scope="module")
def C():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_13651_gb300 import build, clamp
    build.build()
    clamp.load()
    return clamp


class Net:
    """Zero parameters, with views of every layer's weights and biases."""

    def __init__(self, ch):
        self.flat, self.W, self.b, self.at, off = np.zeros(U.param_count(*ch), np.float32), [], [], [], 0
        for kind, ci, co in U.layer_specs(*ch):
            shape = (co, ci, 27) if kind == "conv3" else (ci, co, 8) if kind == "tconv" else (co, ci)
            nw = int(np.prod(shape))
            self.at.append(slice(off, off + nw))
            self.W.append(self.flat[off:off + nw].reshape(shape))
            self.b.append(self.flat[off + nw:off + nw + co])
            off += nw + co


def shifts(w, ci):
    """Output channel c copies input channel ci at tap c mod 27, halved once per 27 channels."""
    for c in range(w.shape[0]):
        w[c, ci, c % 27] = 0.5 ** (c // 27)


def shifted(v, channels):
    """[B][nz][ny][nx] -> [B][channels][..]: what shifts() makes of it."""
    p, (nz, ny, nx) = F.pad(v, (1,) * 6), v.shape[1:]
    return torch.stack([0.5 ** (c // 27) * p[:, c % 27 // 9:, c % 9 // 3:, c % 3:][:, :nz, :ny, :nx]
                        for c in range(channels)], 1)


def exact_wgrad(x, g):
    """FP64 sums over samples and voxels of g[co][v] x[ci][v + tap]."""
    out = torch.zeros(g.shape[1], x.shape[1], 27, dtype=torch.float64, device=x.device)
    for xb, gb in zip(x, g):
        p, gm, (nz, ny, nx) = F.pad(xb.double(), (1,) * 6), gb.double().flatten(1), xb.shape[1:]
        for t in range(27):
            out[:, :, t] += gm @ p[:, t // 9:, t // 3 % 3:, t % 3:][:, :nz, :ny, :nx].flatten(1).t()
    return out


def bf16(v):
    return v.to(torch.bfloat16).to(torch.float32)


def image(B, shape, seed):
    rng = torch.Generator(device="cuda").manual_seed(seed)
    x = bf16(0.5 + 1.5 * torch.rand((B,) + shape, generator=rng, device="cuda"))
    return x, torch.randint(0, 2, x.shape, generator=rng, device="cuda").float() * 2 - 1   # +-1


def run(C, ch, net, layer, x, target, on):
    u = C.UNet(*ch, params=net.flat, dtype="bf16")
    u.set_tensor_cores(on)
    u.backward(x, target, torch.zeros((), dtype=torch.float64, device="cuda"))
    u.check()
    return torch.from_numpy(u.get("grads")[net.at[layer]]).cuda().double()


def error(got, ref):
    return float((got - ref.flatten()).norm() / ref.norm())


# Tensor cores: eight MMAs per chain, each losing up to 2.5e-8 of the sum so far (two thirds of the
# chain's on the average: 1.3e-7 of it, signs at random between chains; the second chain of a pair starts
# from the first's sum: x 1.2), and the FP32 sums of the chains (5e-8): below 2e-7.  CUDA cores: the
# bound that the choice between the two is made for, 2e-5.
TC, CC = 2e-7, 2e-5


# The full-size level, 16 -> 16 channels: 38 shares, so the limit of 24 k terms lies between 28 and 29 samples of
# 32^3.  (nz, ny, nx), samples, on the tensor cores.
@pytest.mark.parametrize("shape,B,on_tc", [((4, 4, 4), 2, False), ((16, 16, 16), 2, True), ((4, 20, 24), 3, True),
                                           ((8, 68, 40), 2, True), ((12, 36, 12), 5, True), ((32, 32, 32), 28, True),
                                           ((32, 32, 32), 29, False)])
def test_full_size_level(C, shape, B, on_tc):
    ch, layer = (16, 4, 4), 11
    net = Net(ch)
    net.W[0][0, 0, 13] = net.W[1][0, 0, 13] = 1       # s1[0] = the image
    shifts(net.W[10], ch[0])
    net.b[11][:] = 1                                  # conv 11's outputs are 1 whatever comes in
    net.W[12][0] = 0.5 ** (np.arange(ch[0]) % 3)
    x, d = image(B, shape, 5)
    target = float(net.W[12].sum()) - d               # output - target = d
    ref = exact_wgrad(shifted(x, ch[0]), bf16(2 * d / x.numel())[:, None] * torch.from_numpy(net.W[12][0]).cuda().view(-1, 1, 1, 1))
    tc, cc = error(run(C, ch, net, layer, x, target, True), ref), error(run(C, ch, net, layer, x, target, False), ref)
    assert tc < (TC if on_tc else CC), (tc, cc)
    assert cc < CC, (tc, cc)


# The half-size level, 64 -> 64 channels: three shares, so the limit of 112 k terms lies between 20 and 22 samples of
# 64x64x32 (327 k and 360 k voxels at half size).
@pytest.mark.parametrize("shape,B,on_tc", [((8, 8, 8), 3, False), ((12, 20, 28), 2, True), ((16, 72, 16), 2, True),
                                           ((32, 64, 64), 20, True), ((32, 64, 64), 22, False)])
def test_half_size_level(C, shape, B, on_tc):
    ch, layer = (4, 64, 4), 8
    net = Net(ch)
    net.W[0][0, 0, 13] = net.W[1][0, 0, 13] = 1       # s1[0] = the image
    net.W[2][0, 0, 13] = net.W[3][0, 0, 13] = 1       # s2[0] = its maxima over 2^3
    shifts(net.W[7], ch[1])
    net.b[8][:] = 1                                   # conv 8's outputs are 1 whatever comes in
    sign = np.where(np.random.default_rng(1).integers(0, 2, (ch[1], 8)) > 0, 1, -1)
    net.W[9][:, 0] = sign
    net.b[9][0] = 128                                 # 64 + 128 at most and at least: above zero, exact in BF16
    net.W[10][0, 0, 13] = net.W[11][0, 0, 13] = 1
    net.W[12][0, 0] = 1
    x, d = image(B, shape, 6)
    nz, ny, nx = shape
    out = torch.from_numpy((128 + sign.sum(0)).reshape(2, 2, 2).astype(np.float32)).cuda()
    target = out.repeat(nz // 2, ny // 2, nx // 2)[None] - d
    pooled = F.max_pool3d(x[:, None], 2)[:, 0]
    child = bf16(2 * d / x.numel()).reshape(B, nz // 2, 2, ny // 2, 2, nx // 2, 2).permute(0, 1, 3, 5, 2, 4, 6).flatten(4)
    g = bf16((child @ torch.from_numpy(sign.T.astype(np.float32)).cuda()).permute(0, 4, 1, 2, 3))   # k times one value, |k| <= 8
    ref = exact_wgrad(shifted(pooled, ch[1]), g)
    tc, cc = run(C, ch, net, layer, x, target, True), run(C, ch, net, layer, x, target, False)
    assert error(cc, ref) < CC
    if on_tc:
        assert error(tc, ref) < TC
    else:   # the same kernel: its three shares in another order at most (a few times 2^-24)
        assert float((tc - cc).norm() / ref.norm()) < TC
