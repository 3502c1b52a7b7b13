"""The start-vector network on grids at the edges of its convolution and
weight-gradient tiles (32 x 8 and 16 x 8 pixels, one kernel for large grids and
one for small ones), against the FP64 oracle with the FP16-rounded weights.

Bounds as for the other grids: forward 1e-4 of the output's scale, gradients
1e-3 relative as a whole and per layer (FP32 sums of at most 288 products per
output and 4e4 per weight stay far inside; a missed or repeated row, column
or tile does not).
"""
import numpy as np
import pytest

from oracle import warmstart as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Wd", [(8, 8), (24, 72), (4872, 8), (72, 264)])
def test_forward_and_gradient_at_tile_edges(H, Wd):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_05400_gb300 import build as B
    B.build()
    from paper_2508_05400_gb300 import rks
    rng = np.random.default_rng(H + Wd)
    x = rng.standard_normal((3, H, Wd)).astype(np.float32)
    Q = np.linalg.qr(rng.standard_normal((H * Wd, 3)))[0].astype(np.float32)
    with rks.WarmStart(H, Wd, seed=9) as net:
        theta = net.params()
        xd = torch.from_numpy(x).cuda()
        u = net.forward(xd).cpu().numpy()
        net.accumulate(xd, torch.from_numpy(np.ascontiguousarray(Q.T)).cuda())
        g = net.grad().astype(np.float64)
    th, o = theta.astype(np.float64), 0
    for i, sz in enumerate(W.param_sizes()):
        if i % 2 == 0:
            th[o:o + sz] = theta[o:o + sz].astype(np.float16).astype(np.float64)
        o += sz
    uo, _ = W.forward(th, x.astype(np.float64))
    assert np.max(np.abs(u - uo)) <= 1e-4 * np.max(np.abs(uo))
    _, go, _ = W.loss_and_grad(th, x.astype(np.float64), Q.astype(np.float64))
    assert np.linalg.norm(g - go) <= 1e-3 * np.linalg.norm(go)
    o = 0
    for i, sz in enumerate(W.param_sizes()):
        a, b = g[o:o + sz], go[o:o + sz]
        assert np.linalg.norm(a - b) <= 1e-3 * np.linalg.norm(b) + 1e-7 * np.linalg.norm(go), i
        o += sz
