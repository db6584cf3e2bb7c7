"""The U-Net's tensor-core 3x3x3 conv at the edges of its tiles (32 or 16 x voxels, 16 rows, up to
8 planes, 304 persistent CTAs): heights below and beside 16 rows, plane counts that do not
fill a tile, one tile and several per CTA."""
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


# Both paths round the same operands to BF16; only the order of the FP32 sums differs, and a
# rounding flip grows through the layers to at most about 1e-2 (tests/test_gpu_unet_tc.py
# uses 1.5e-2 for the same comparison).  A voxel that a tile missed or wrote twice is of order 1
# locally, so the largest difference is bounded too.
@pytest.mark.parametrize("shape,B", [((4, 4, 32), 1), ((12, 20, 64), 2), ((8, 8, 16), 3), ((20, 36, 128), 1),
                                     ((4, 40, 96), 5), ((52, 16, 32), 2), ((36, 72, 64), 9)])
def test_forward_matches_cuda_cores(C, shape, B):
    ch = (16, 32, 64)
    p = I.unet_params(ch, seed=31)
    p[-1] = 0.5
    x = torch.rand((B,) + shape, generator=torch.Generator(device="cuda").manual_seed(32), device="cuda") * 2
    out = []
    for on in (True, False):
        net = C.UNet(*ch, params=p, dtype="bf16")
        net.set_tensor_cores(on)
        out.append(net.forward(x).cpu().numpy().astype(np.float64))
        net.check()
    tc, cc = out
    assert np.isfinite(tc).all()
    assert np.linalg.norm(tc - cc) < 1.5e-2 * np.linalg.norm(cc)
    assert np.abs(tc - cc).max() < 0.25 * np.sqrt(np.mean(cc * cc))
