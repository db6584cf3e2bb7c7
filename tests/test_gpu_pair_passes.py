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
