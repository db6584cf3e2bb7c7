"""The U-Net's CUDA-core 3x3x3 conv with eight x voxels per thread, which large levels take: 16 and 32 wide tiles
with 16, 32 and 64 output channels, rows that end inside a tile, channels that leave part of a block unused.  Many copies of one sample
make the level large; every copy is compared with the oracle's single output."""
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


# Eight voxels from 152 x 8 x 32 x 64 outputs on.  Widths (tile, channels) of the levels: 36 (16, 16), 18 (32, 32),
# 9 (16, 64 + 8); 60 (32, 33 of 64), 30 (32, 16), 15 (16, 24 of 32); 40 (16, 20 of 32), 20 (32, 48 of 64).
# Bounds as for the other FP32 forward passes (ten layers of at most 27 x 72 terms).
@pytest.mark.parametrize("ch,shape,B", [((16, 32, 72), (4, 12, 36), 1500), ((33, 16, 24), (4, 12, 60), 2400),
                                        ((20, 48, 4), (4, 12, 40), 300)])
def test_forward_matches_oracle(C, ch, shape, B):
    n = int(np.prod(shape))
    assert all(B * n // d * c >= 152 * 8 * 32 * 64 for c, d in zip(ch, (1, 8, 64)) if c != 4)
    p = I.unet_params(ch, seed=51)
    p[-1] = 0.5
    x = np.random.default_rng(52).uniform(0.0, 2.0, size=(1,) + shape).astype(np.float32)
    net = C.UNet(*ch, params=p, dtype="fp32")
    got = net.forward(torch.from_numpy(x).cuda().expand(B, *shape).contiguous()).double()
    ref = U.forward(p.astype(np.float64), x.astype(np.float64), ch).cuda()
    err = (got - ref).flatten(1)
    assert float(err.norm(dim=1).max()) < 1e-5 * float(ref.norm())
    assert float(err.abs().max()) < 1e-3 * float(ref.square().mean().sqrt())
