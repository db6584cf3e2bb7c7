"""The transposed convs forward at the edges of their runs (128 or 64 voxels): samples that are no
whole runs or groups of four voxels, more input channels than two buffers hold, several runs."""
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


# FP32 network against exact arithmetic, 1e-5 as for the other FP32 forward tests
@pytest.mark.parametrize("ch,shape,B", [((4, 8, 16), (4, 4, 12), 3), ((4, 20, 36), (20, 36, 44), 2), ((4, 4, 80), (12, 20, 28), 2),
                                        ((4, 80, 8), (8, 20, 36), 1), ((16, 32, 64), (8, 64, 64), 1)])
def test_forward_matches_oracle(C, ch, shape, B):
    p = I.unet_params(ch, seed=71)
    p[-1] = 0.5
    x = np.random.default_rng(72).uniform(0.0, 2.0, size=(B,) + shape).astype(np.float32)
    net = C.UNet(*ch, params=p, dtype="fp32")
    got = net.forward(torch.from_numpy(x).cuda()).cpu().numpy().astype(np.float64)
    ref = U.forward(p.astype(np.float64), x.astype(np.float64), ch).numpy()
    assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)
    assert np.abs(got - ref).max() < 1e-3 * np.sqrt(np.mean(ref * ref))
