"""Inference of many rows runs in passes over a bounded workspace that holds nothing of
the gradient's, and the passes change no bit of a row's result."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_in,H,rows", [(2048, 64, 1 << 17), (13, 128, 1 << 18), (13, 128, (1 << 18) + 65),
                                         (40, 1500, 100001)])
def test_inference_workspace(n_in, H, rows):
    import paper_2006_02501_gb300 as mh
    net = mh.MLP(n_in, H, 6, seed=3)
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((rows, n_in), generator=g, device="cuda")
    y = torch.zeros((rows, 6), device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    net.forward(x, y)
    torch.cuda.synchronize()
    held = free - torch.cuda.mem_get_info()[0]
    assert held < 320 << 20, held              # 256 MB and allocation granules
    assert torch.isfinite(y).all()
    for a, b in ((0, 777), (rows // 2 - 5, rows // 2 + 400), (rows - 301, rows)):
        part = torch.zeros((b - a, 6), device="cuda")
        net.forward(x[a:b].contiguous(), part)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(part.cpu().numpy(), y[a:b].cpu().numpy())
    # the gradient's pass takes its buffers beside the inference's, in either order
    t = torch.randn((500, 6), generator=g, device="cuda")
    loss, grad = net.loss_grad(x[:500].contiguous(), t)
    other = mh.MLP(n_in, H, 6, seed=3)
    loss2, grad2 = other.loss_grad(x[:500].contiguous(), t)
    assert loss == loss2
    np.testing.assert_array_equal(grad, grad2)
    net.close()
    other.close()
