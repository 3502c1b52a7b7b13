"""The start-vector network on grids at the edges of its convolution and
weight-gradient tiles (32 x 8 and 16 x 8 pixels, one kernel for large grids and
one for small ones), against the FP64 oracle with the FP16-rounded weights.

The gradients are taken of a network whose ReLU inputs are all far from zero
(small weights, unit biases): an input within FP32 rounding of zero may fall
on the other side in FP64, which moves the gradient of an incoherent target
by far more than the kernels' rounding.  Bounds as for the other grids:
forward 1e-4 of the output's scale, gradients 1e-3 relative as a whole and per
layer (FP32 sums of at most 288 products per output and 4e4 per weight stay
far inside; a missed or repeated row, column or tile does not).
"""
import numpy as np
import pytest

from oracle import warmstart as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_05400_gb300 import build as B
    B.build()
    return torch


def _fp16_weights(theta):
    th, o = theta.astype(np.float64), 0
    for i, sz in enumerate(W.param_sizes()):
        if i % 2 == 0:
            th[o:o + sz] = theta[o:o + sz].astype(np.float16).astype(np.float64)
        o += sz
    return th


def _sample(H, Wd):
    rng = np.random.default_rng(H + Wd)
    x = rng.standard_normal((3, H, Wd)).astype(np.float32)
    return x, np.linalg.qr(rng.standard_normal((H * Wd, 3)))[0].astype(np.float32)


SIZES = [(8, 8), (24, 72), (4872, 8), (72, 264)]


@pytest.mark.parametrize("H,Wd", SIZES)
def test_forward_at_tile_edges(gpu, H, Wd):
    from paper_2508_05400_gb300 import rks
    x, _ = _sample(H, Wd)
    with rks.WarmStart(H, Wd, seed=9) as net:
        theta = net.params()
        u = net.forward(gpu.from_numpy(x).cuda()).cpu().numpy()
    uo, _ = W.forward(_fp16_weights(theta), x.astype(np.float64))
    assert np.max(np.abs(u - uo)) <= 1e-4 * np.max(np.abs(uo))


@pytest.mark.parametrize("H,Wd", SIZES)
def test_gradient_at_tile_edges_with_every_unit_active(gpu, H, Wd):
    from paper_2508_05400_gb300 import rks
    x, Q = _sample(H, Wd)
    with rks.WarmStart(H, Wd, seed=9) as net:
        theta, o = net.params(), 0
        for i, sz in enumerate(W.param_sizes()):
            theta[o:o + sz] = theta[o:o + sz] * 0.1 if i % 2 == 0 else 1.0
            o += sz
        net.set_params(theta)
        net.accumulate(gpu.from_numpy(x).cuda(), gpu.from_numpy(np.ascontiguousarray(Q.T)).cuda())
        g = net.grad().astype(np.float64)
    _, go, _ = W.loss_and_grad(_fp16_weights(theta), x.astype(np.float64), Q.astype(np.float64))
    assert np.linalg.norm(g - go) <= 1e-3 * np.linalg.norm(go)
    o = 0
    for i, sz in enumerate(W.param_sizes()):
        a, b = g[o:o + sz], go[o:o + sz]
        assert np.linalg.norm(a - b) <= 1e-3 * np.linalg.norm(b) + 1e-7 * np.linalg.norm(go), i
        o += sz
