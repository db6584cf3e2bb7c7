"""The warm start's scaling by the mean per column: aligned and unaligned inputs, sums that FP32 does
not hold, sizes with fewer groups of four than threads."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_13651_gb300 import inputs as I  # noqa: E402


@pytest.fixture(scope="module")
def C():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_13651_gb300 import build, clamp
    build.build()
    clamp.load()
    return clamp


# U(x / m) with m = sum(x) / (nx ny): scaling x by a power of two scales the result by it exactly, also
# where four values' FP32 sum would overflow (2^126: the sums go to FP64 one by one there); an
# unaligned input takes the scalar kernels, whose m differs by FP64 rounding: one FP32 step of each
# value, which the BF16 network may turn into a rounding flip (1.5e-2, as between its conv paths).
@pytest.mark.parametrize("shape", [(4, 4, 4), (8, 12, 20), (16, 64, 96)])
def test_scaling_and_alignment(C, shape):
    p = I.unet_params((4, 8, 16), seed=91)
    net = C.UNet(4, 8, 16, params=p, dtype="bf16")
    x = torch.rand(shape, generator=torch.Generator(device="cuda").manual_seed(92), device="cuda") + 0.5
    ref = net.warm_start(x, 1e-3).double()
    assert torch.isfinite(ref).all()
    for e in (-90, 60, 100):
        got = net.warm_start(x * 2.0 ** e, 1e-3).double()
        assert torch.equal(got, ref * 2.0 ** e)
    buf = torch.empty(x.numel() + 1, device="cuda")
    v = buf[1:].view(shape)
    v.copy_(x)
    got = net.warm_start(v, 1e-3).double()
    assert float((got - ref).norm()) < 1.5e-2 * float(ref.norm())


def test_values_near_the_largest(C):
    """Four values whose FP32 sum overflows: the sum is taken in FP64."""
    p = I.unet_params((4, 8, 16), seed=91)
    net = C.UNet(4, 8, 16, params=p, dtype="bf16")
    x = torch.zeros((4, 4, 4), device="cuda")
    x[0] = 2.0 ** 127   # m = 2^127
    y = torch.zeros((4, 4, 4), device="cuda")
    y[0] = 1.0          # m = 1
    a, b = net.warm_start(x, 1e-3), net.warm_start(y, 1e-3)
    big = b.double() * 2.0 ** 127
    ok = big < 3.4e38
    assert torch.equal(a.double()[ok], big[ok])
