"""The set-up passes (simulation, back-projection) at every transform length on every axis,
against double-precision FFTs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_13651_gb300 import build, clamp
    build.build()
    clamp.load()
    return clamp


# FP32 transforms of up to 24 radix-2 stages' depth, about 1e-7 each way: 1e-6
@pytest.mark.parametrize("shape", [(8, 8, 16), (16, 256, 32), (32, 16, 64), (64, 192, 96), (96, 32, 128), (128, 64, 192),
                                   (192, 96, 16), (256, 128, 16), (16, 16, 256)])
def test_simulate_and_back_projection(C, shape):
    nz, ny, nx = shape
    L, nv = 2, 0.01
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    cn = lambda: torch.view_as_complex(torch.randn((L,) + shape + (2,), generator=g, device="cuda"))
    r = torch.rand(shape, generator=g, device="cuda")
    z, eta = cn(), cn()
    pupil = torch.rand((ny, nx), generator=g, device="cuda") * (torch.rand((ny, nx), generator=g, device="cuda") < 0.3)
    window = torch.rand((nz,), generator=g, device="cuda")
    a = window.double()[:, None, None] * pupil.double()[None]
    p = C.make_params(nx, ny, nz, L, nv, 1e-4)
    y = C.simulate(p, r, z, eta, pupil, window)
    ref = a * torch.fft.fftn(r.double().sqrt() * z.to(torch.complex128), dim=(1, 2, 3), norm="ortho") \
        + np.sqrt(np.float64(np.float32(nv))) * eta.to(torch.complex128)
    assert float((y - ref).norm()) < 1e-6 * float(ref.norm())
    mu, _, _ = C.init(p, y, pupil, window)
    ref = torch.fft.ifftn(a * y.to(torch.complex128), dim=(1, 2, 3), norm="ortho") / a.square().mean()
    assert float((mu - ref).norm()) < 1e-6 * float(ref.norm())
