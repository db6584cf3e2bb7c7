"""A volume whose rows of tiles are more than a grid's y extent: 262148 rows, 33 channels."""
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


def test_tall_volume(C):
    nx, ny, nz, crop, seen = 20, 262148, 4, 128, 64
    net = C.UNet(33, 2, 2, params=I.unet_params((33, 2, 2), seed=2), dtype="fp32")
    rng = torch.Generator(device="cuda").manual_seed(1)
    x = torch.rand((1, nz, ny, nx), generator=rng, device="cuda")
    y = net.forward(x)
    # rows further than the receptive field (22 rows) from a crop's cut edge see the same inputs; the same FP32
    # chains whatever the tiles
    top, bottom = net.forward(x[:, :, :crop].contiguous()), net.forward(x[:, :, ny - crop:].contiguous())
    assert torch.isfinite(y).all() and float(y.std()) > 0
    np.testing.assert_allclose(y[:, :, :seen].cpu(), top[:, :, :seen].cpu(), rtol=1e-6, atol=1e-7)
    np.testing.assert_allclose(y[:, :, ny - seen:].cpu(), bottom[:, :, crop - seen:].cpu(), rtol=1e-6, atol=1e-7)
