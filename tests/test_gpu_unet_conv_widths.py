"""The U-Net's CUDA-core 3x3x3 conv at the edges of its tiles (8, 16 or 32 x voxels, 4 to 16
rows, 16, 32 or 64 output channels): widths below, at and beside each tile width, rows that
are no multiple of four, channel counts that leave part of a block unused, several blocks."""
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


# FP32 sums of at most 27 x 72 terms per output, ten layers: the largest chain's worst case is
# 2000 x 6e-8 = 1.2e-4, its random-sign size about 3e-6; 1e-5 as for the other FP32 networks.
@pytest.mark.parametrize("ch,shape,B", [((4, 8, 16), (4, 4, 4), 1), ((5, 12, 36), (4, 20, 12), 2),
                                        ((16, 32, 64), (8, 36, 32), 1), ((16, 32, 72), (4, 8, 68), 1),
                                        ((3, 17, 33), (8, 12, 60), 3)])
def test_forward_matches_oracle(C, ch, shape, B):
    p = I.unet_params(ch, seed=41)
    p[-1] = 0.5
    x = np.random.default_rng(42).uniform(0.0, 2.0, size=(B,) + shape).astype(np.float32)
    net = C.UNet(*ch, params=p, dtype="fp32")
    got = net.forward(torch.from_numpy(x).cuda()).cpu().numpy().astype(np.float64)
    ref = U.forward(p.astype(np.float64), x.astype(np.float64), ch).numpy()
    assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)
    # one voxel missed or written twice is of order 1 there
    assert np.abs(got - ref).max() < 1e-3 * np.sqrt(np.mean(ref * ref))
