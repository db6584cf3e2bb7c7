"""The support tables of the band-limited schedule, the vectorised element-wise passes against the scalar kernels that take unaligned arrays, and
the Gaussian prior agent's marching kernel at the edges of its columns and plane blocks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import clamp_oracle as O  # noqa: E402
from paper_2406_13651_gb300 import inputs as I  # noqa: E402


@pytest.fixture(scope="module")
def C():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_13651_gb300 import build, clamp
    build.build()
    clamp.load()
    return clamp


def _off_by_one(t):
    """A copy of t that starts one element past an aligned address."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = buf[1:].view(t.shape)
    v.copy_(t)
    return v


# 27 FMAs of positive terms with weights that sum to 1: 27 x 6e-8 = 1.6e-6 at most
@pytest.mark.parametrize("shape", [(1, 1, 4), (2, 3, 8), (5, 7, 12), (3, 5, 6), (40, 9, 100), (33, 31, 256), (17, 2, 1024)])
def test_gauss_matches_oracle(C, shape):
    x = torch.rand(shape, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    den = C.Denoiser.gauss(0.8)
    out, scalar = torch.empty_like(x), torch.empty_like(x)
    C.denoise(den, x, out)
    C.denoise(den, _off_by_one(x), scalar)
    ref = O.denoise_gauss(x.cpu().numpy().astype(np.float64), 0.8)
    assert np.abs(out.cpu().numpy() - ref).max() < 2e-6
    assert torch.equal(out, scalar)


# the same arithmetic per voxel: equal bits.  The convergence error's FP32 partial sums run in
# another order: at most a few hundred positive terms each, 1e-5 of the sum.
@pytest.mark.parametrize("L", [1, 2, 3, 9, 17])
@pytest.mark.parametrize("shape", [(16, 8, 8), (32, 96, 16)])
def test_pair_passes_match_scalar_passes(C, shape, L):
    nx, ny, nz = shape
    wl = I.make_workload("cfg1", seed=5, nx=nx, ny=ny, nz=nz, looks=L, iters=1)
    p = C.make_params(nx, ny, nz, L, wl.noise_var, 1e-3, max_iters=1)
    g = torch.Generator(device="cuda").manual_seed(6)
    y = torch.view_as_complex(torch.randn((L, nz, ny, nx, 2), generator=g, device="cuda"))
    mu = torch.view_as_complex(torch.randn((L, nz, ny, nx, 2), generator=g, device="cuda"))
    r = torch.rand((L + 1, nz, ny, nx), generator=g, device="cuda") + 0.05
    w = torch.rand((L + 1, nz, ny, nx), generator=g, device="cuda") + 0.05
    pupil, window = torch.from_numpy(wl.pupil).cuda(), torch.from_numpy(wl.window).cuda()
    got = []
    for f in (torch.clone, _off_by_one):
        m, rr, ww, ce = f(mu), f(r), f(w), torch.zeros(1, dtype=torch.float64, device="cuda")
        wbar = f(r[0])
        C.forward_prox(p, 3, y, pupil, window, m, rr, ww)
        C.mace_step(p, rr, ww, wbar, ce)
        got.append((m, rr, ww, wbar, float(ce.item())))
    for a, b in zip(got[0][:4], got[1][:4]):
        assert torch.isfinite(torch.view_as_real(a) if a.is_complex() else a).all()
        assert torch.equal(a, b)
    assert abs(got[0][4] - got[1][4]) <= 1e-5 * got[1][4]


# one support point at a time through the tables' 32-column words and row blocks: the
# band-limited and the full-spectrum schedule give the same step
@pytest.mark.parametrize("nx,ny", [(16, 8), (32, 64), (96, 32), (192, 16), (256, 256)])
@pytest.mark.parametrize("fill", [0.003, 0.15])
def test_band_tables_of_ragged_pupils(C, nx, ny, fill):
    rng = np.random.default_rng(nx + ny)
    pupil = ((rng.uniform(size=(ny, nx)) < fill) * rng.uniform(0.5, 1.0, (ny, nx))).astype(np.float32)
    pupil[0, 0] = pupil[ny - 1, nx - 1] = 0.75
    L, nz = 2, 8
    wl = I.make_workload("cfg1", seed=7, nx=nx, ny=ny, nz=nz, looks=L, iters=1)
    g = torch.Generator(device="cuda").manual_seed(8)
    y = torch.view_as_complex(torch.randn((L, nz, ny, nx, 2), generator=g, device="cuda"))
    mu = torch.view_as_complex(torch.randn((L, nz, ny, nx, 2), generator=g, device="cuda"))
    r = torch.rand((L + 1, nz, ny, nx), generator=g, device="cuda") + 0.05
    got = []
    for flag in (C.FLAG_BAND_SPECTRUM, C.FLAG_FULL_SPECTRUM):
        p = C.make_params(nx, ny, nz, L, wl.noise_var, 1e-3, max_iters=1)
        p.flags |= flag
        m, rr = mu.clone(), r.clone()
        C.forward_prox(p, 3, y, torch.from_numpy(pupil).cuda(), torch.from_numpy(wl.window).cuda(), m, rr, r.clone())
        got.append((torch.view_as_real(m).double().cpu(), rr.double().cpu()))
    for a, b in zip(*got):   # FP32 transforms of about 20 stages on both sides, as for the oracle comparisons
        assert float((a - b).norm()) < 1e-5 * float(b.norm())
