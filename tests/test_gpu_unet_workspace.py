"""The U-Net's entry points refuse a workspace that is not 256-byte aligned before any launch."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_misaligned_workspace_is_refused():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_13651_gb300 import build, clamp as C
    build.build()
    lib, net, B, n = C.load(), C.UNet(4, 8, 16, dtype="bf16"), 2, 8
    x, y = (torch.ones((B, n, n, n), device="cuda") for _ in range(2))
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    size = lib.clamp_unet_workspace_size(net.handle, B, n, n, n, 1)
    buf = torch.empty(size + 512, dtype=torch.uint8, device="cuda")
    base = (buf.data_ptr() + 255) // 256 * 256
    P = lambda t: t.data_ptr()   # noqa: E731

    def calls(ws):
        return [lib.clamp_unet_forward(net.handle, P(x), P(y), B, n, n, n, ws, size, None),
                lib.clamp_unet_backward(net.handle, P(x), P(y), B, n, n, n, P(loss), ws, size, None),
                lib.clamp_unet_loss(net.handle, P(x), P(y), B, n, n, n, P(loss), ws, size, None),
                lib.clamp_unet_warm_start(net.handle, n, n, n, P(x), 1e-3, P(y), ws, size, None)]

    for off in (4, 8, 16, 128):
        assert calls(base + off) == [1] * 4, off      # CLAMP_EINVAL
    assert calls(base) == [0] * 4
    torch.cuda.synchronize()
