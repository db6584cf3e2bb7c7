"""The transposed convs' weight gradient over many chunks per CTA: its register sums are
flushed every eight chunks, and a CTA's share need not be whole samples."""
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


# The loss is a mean over the batch, so B copies of a sample have its gradient: every sum runs
# over B times as many terms and any missed, doubled or misplaced chunk shows.  FP32 sums in
# chains of at most a few thousand terms: 1e-5.
@pytest.mark.parametrize("ch,shape,B", [((16, 32, 64), (16, 64, 64), 48), ((4, 20, 36), (12, 20, 36), 100),
                                        ((8, 8, 8), (4, 4, 4), 1000)])
def test_copies_of_a_sample_keep_its_gradient(C, ch, shape, B):
    p = I.unet_params(ch, seed=51)
    p[-1] = 0.5
    g = torch.Generator(device="cuda").manual_seed(52)
    x, t = (torch.rand((1,) + shape, generator=g, device="cuda") for _ in range(2))
    grads = []
    for n in (1, B):
        net = C.UNet(*ch, params=p, dtype="fp32")
        loss = torch.zeros((), dtype=torch.float64, device="cuda")
        net.backward(x.expand((n,) + shape).contiguous(), t.expand((n,) + shape).contiguous(), loss)
        grads.append(net.get("grads").astype(np.float64))
    off = 0
    for kind, ci, co in U.layer_specs(*ch):
        nw = co * ci * (27 if kind == "conv3" else 8 if kind == "tconv" else 1)
        if kind == "tconv":
            a, b = grads[0][off:off + nw], grads[1][off:off + nw]
            assert np.linalg.norm(a) > 0
            assert np.linalg.norm(a - b) < 1e-5 * np.linalg.norm(a)
        off += nw + co
