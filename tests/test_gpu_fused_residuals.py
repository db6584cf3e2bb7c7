"""The line search and the residuals formed by the last CTA of their passes: one and many CTAs
per look, one and many looks, several iterations in one call (the counters return to zero)."""
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


# The convergence error of iteration k from its definition in FP64 on the states before and after
# it: FP32 partial sums of positive terms, 1e-5.
@pytest.mark.parametrize("schedule", ["FLAG_BAND_SPECTRUM", "FLAG_FULL_SPECTRUM"])
@pytest.mark.parametrize("shape,L", [((16, 8, 8), 1), ((32, 32, 16), 4), ((64, 96, 8), 33), ((128, 64, 64), 3)])
def test_convergence_error_of_every_iteration(C, shape, L, schedule):
    nx, ny, nz = shape
    wl = I.make_workload("cfg1", seed=9, nx=nx, ny=ny, nz=nz, looks=L, iters=1)
    p = C.make_params(nx, ny, nz, L, wl.noise_var, 1e-3)
    p.flags |= getattr(C, schedule)
    g = torch.Generator(device="cuda").manual_seed(10)
    cn = lambda: torch.view_as_complex(torch.randn((L, nz, ny, nx, 2), generator=g, device="cuda"))
    y, mu = cn(), cn()
    r = (torch.rand((nz, ny, nx), generator=g, device="cuda") + 0.05).expand(L + 1, nz, ny, nx).contiguous()
    w, wbar = r.clone(), torch.empty_like(r[0])
    pupil, window = torch.from_numpy(wl.pupil).cuda(), torch.from_numpy(wl.window).cuda()
    den = C.Denoiser.gauss(0.8)
    ws = C.iterate_workspace(p, den)
    n, ups = 6, torch.full((L + 1,), (1.0 - p.prior_weight) / L, dtype=torch.float64, device="cuda")
    ups[L] = p.prior_weight
    a = [mu.clone(), r.clone(), w.clone()]
    ref = []
    for k in range(n):   # one iteration per call, the error from the states around it
        before = (ups[:, None, None, None] * a[2].double()).sum(0)
        C.iterate(p, 1 + k, 1, y, pupil, window, den, a[0], a[1], a[2], wbar, ws=ws)
        num = (a[1].double() - before[None]).square().sum()
        ref.append(float((num / ((L + 1) * before.square().sum())).sqrt()))
    ce = torch.zeros(n, dtype=torch.float64, device="cuda")
    for _ in range(2):   # all in one call, twice on the same workspace
        b = [mu.clone(), r.clone(), w.clone()]
        C.iterate(p, 1, n, y, pupil, window, den, b[0], b[1], b[2], wbar, ce_out=ce, ws=ws)
        got = ce.cpu().numpy()
        # the spectrum advanced by gamma F d instead of formed afresh: FP32 rounding of the state
        np.testing.assert_allclose(got, ref, rtol=1e-4)
        assert abs(got[0] - ref[0]) <= 1e-5 * ref[0]
