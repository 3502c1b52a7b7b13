"""The start-vector network on a grid of more than 65 535 convolution tiles in
height.  Its receptive field is local (three poolings, 15 convolutions: fewer
than 128 rows), so the first rows are those of the same network on a short
grid with the same first rows, and the last ones those of one with the same
last rows, bit for bit: the sums are formed in the same order.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_05400_gb300 import build as B
    B.build()
    return torch


def test_tall_grid(gpu):
    from paper_2508_05400_gb300 import rks
    H, W, h = 8 * 65_535 + 64, 8, 1024
    g = gpu.Generator().manual_seed(3)
    x = gpu.randn(3, H, W, generator=g).cuda()
    q = gpu.randn(1, H * W, generator=g).cuda() / (H * W) ** 0.5
    with rks.WarmStart(H, W, seed=5) as net:
        u = net.forward(x)
        net.zero_grad()
        loss = net.accumulate(x, q)
        grad = net.grad()
    with rks.WarmStart(h, W, seed=5) as net:
        top, end = net.forward(x[:, :h].contiguous()), net.forward(x[:, H - h:].contiguous())
    assert gpu.equal(u[:h - 128], top[:h - 128]) and gpu.equal(u[H - h + 128:], end[128:])
    assert 0.0 <= loss <= 1.0 and abs(grad).max() > 0.0 and abs(grad).max() < 1e6
