"""The transposed convs' data gradient with four voxels per thread (many runs) and one (few), at
samples that are no whole runs: gradients of the layers below it against the oracle's."""
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


# B copies of a sample have its mean gradient, whatever path their number takes.  The first layer's
# weights see every data gradient, and its FP32 sums run in chains of at most 7 k terms (one input
# channel: 608 / ceil(channels / 16) shares of the volume), so 1e-5.  Deeper layers' sums are not
# compared: with one share for 264 input channels their chains are 300 k terms long.
@pytest.mark.parametrize("ch,shape,B", [((4, 8, 16), (12, 20, 28), 200), ((4, 36, 40), (8, 36, 44), 80), ((4, 132, 8), (4, 12, 20), 320),
                                        ((4, 8, 16), (4, 4, 4), 320)])
def test_few_and_many_runs_agree(C, ch, shape, B):
    p = I.unet_params(ch, seed=81)
    p[-1] = 0.5
    g = torch.Generator(device="cuda").manual_seed(82)
    x, t = (torch.rand((1,) + shape, generator=g, device="cuda") for _ in range(2))
    grads = []
    for n in (1, B):
        net = C.UNet(*ch, params=p, dtype="fp32")
        loss = torch.zeros((), dtype=torch.float64, device="cuda")
        net.backward(x.expand((n,) + shape).contiguous(), t.expand((n,) + shape).contiguous(), loss)
        grads.append(net.get("grads").astype(np.float64)[:27 * ch[0]])
    a, b = grads
    assert np.linalg.norm(a) > 0
    assert np.linalg.norm(a - b) < 1e-5 * np.linalg.norm(a)
