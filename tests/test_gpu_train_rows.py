"""Widths and batch sizes at the edges of the training step's vector kernels
(column groups of four, grids of whole rows, split sums) against the FP64
oracle's derivative-label gradient, and the loss selection at the ends of its
range."""
import numpy as np
import pytest

import workloads
from oracle import mlp as omlp
from oracle import risk as orisk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import torch
    assert torch.cuda.is_available()
    import paper_1906_02818_gb300 as gb
    return gb


@pytest.mark.parametrize("mode", ["fp32", "tf32x3"])
@pytest.mark.parametrize("width,hidden,n,dirs", [(64, 2, 1, 2), (64, 3, 257, 1), (192, 2, 130, 2), (320, 2, 66, 0),
                                                 (192, 3, 1025, 4), (1024, 2, 33, 1)])
def test_gradient_at_other_widths(gb, mode, width, hidden, n, dirs):
    import torch
    sizes = [5] + [width] * hidden + [1]
    init = workloads.mlp_init(5, width, hidden, seed=3)
    net = gb.Mlp(5, width, hidden, init)
    net.set_train_mode(mode)
    rng = np.random.default_rng(n)
    x = rng.uniform(-1, 1, (n, 5)).astype(np.float32)
    t = rng.uniform(0, 0.5, n).astype(np.float32)
    g = rng.uniform(-1, 1, (n, dirs)).astype(np.float32)
    if n > 8 and dirs:
        g[::5, 0] = np.nan
    d, sc, wt = list(range(dirs)), [1.5, 0.7, 2.0, 1.0][:dirs], [0.5, 2.0, 1.0, 0.3][:dirs]
    parts, grad = net.loss_grad_d(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(),
                                  torch.from_numpy(g).cuda() if dirs else None, d, sc, wt)
    s = np.array(sc)
    loss, p_ref, G = omlp.dloss_and_grads(omlp.unpack(init.astype(np.float64), sizes), x.astype(np.float64),
                                          t.astype(np.float64), g.astype(np.float64) / s if dirs else g.astype(np.float64),
                                          d, list(np.array(wt) * s * s))
    ref = omlp.pack(G)
    assert np.max(np.abs(grad - ref)) <= 1e-4 * np.max(np.abs(ref))
    net.close()


@pytest.mark.parametrize("n,alpha", [(1, 0.5), (2, 0.99), (1023, 0.999), (1024, 0.5), (1025, 0.01), (311_297, 0.99),
                                     (1 << 20, 0.9999)])
def test_loss_selection(gb, n, alpha):
    """Signs, equal losses, infinities and a wide range of exponents."""
    import torch
    rng = np.random.default_rng(n)
    pnl = rng.standard_normal(n) * np.exp(rng.uniform(-40, 40, n))
    pnl[rng.integers(0, n, n // 7)] = 0.0
    if n > 1000:
        pnl[:3] = np.inf
        pnl[5:9] = -0.0
    got = gb.tail(torch.from_numpy(pnl).cuda(), alpha)
    var, cvar, nt = orisk.var_cvar(pnl, alpha)
    assert got["var"] == var and got["n_tail"] == nt, (n, alpha, got, var, nt)
    assert abs(got["cvar"] - cvar) <= 1e-12 * max(1.0, abs(cvar))


@pytest.mark.parametrize("mode", ["fp32", "tf32x3"])
@pytest.mark.parametrize("dirs", [[0, 0], [1, 0, 1], [2, 2, 2, 2], [4, 3, 3, 4]])
def test_directions_that_share_an_input(gb, mode, dirs):
    """Every direction's share of the first layer's gradient arrives where
    several name the same input."""
    import torch
    width, hidden, n, k = 128, 2, 515, len(dirs)
    sizes = [5] + [width] * hidden + [1]
    init = workloads.mlp_init(5, width, hidden, seed=5)
    net = gb.Mlp(5, width, hidden, init)
    net.set_train_mode(mode)
    rng = np.random.default_rng(k)
    x = rng.uniform(-1, 1, (n, 5)).astype(np.float32)
    t = rng.uniform(0, 0.5, n).astype(np.float32)
    g = rng.uniform(-1, 1, (n, k)).astype(np.float32)
    sc, wt = np.array([1.5, 0.7, 2.0, 1.0][:k]), np.array([0.5, 2.0, 1.0, 0.3][:k])
    parts, grad = net.loss_grad_d(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), torch.from_numpy(g).cuda(),
                                  dirs, list(sc), list(wt))
    loss, p_ref, G = omlp.dloss_and_grads(omlp.unpack(init.astype(np.float64), sizes), x.astype(np.float64),
                                          t.astype(np.float64), g.astype(np.float64) / sc, dirs, list(wt * sc * sc))
    ref = omlp.pack(G)
    assert np.max(np.abs(grad - ref)) <= 1e-4 * np.max(np.abs(ref))
    net.close()
