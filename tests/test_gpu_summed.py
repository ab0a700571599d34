"""The kernels that contract a path's summed normals once (European payoffs,
log-Euler) at the widths and step counts where the sums can go wrong: every
residue of d mod 4 (steps that start inside a Philox block), fewer steps than
a segment period, ragged last tiles, against the FP64 oracle."""
import numpy as np
import pytest

from gpu_util import REL, cfg_of, gbm_model, oracle_gbm
from test_gpu_big import _case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import torch
    assert torch.cuda.is_available()
    import paper_1906_02818_gb300 as gb
    return gb


@pytest.mark.parametrize("d,steps,paths", [(65, 1, 65), (66, 2, 130), (67, 3, 64), (68, 5, 63), (126, 4, 100),
                                           (129, 7, 129), (255, 6, 66), (258, 2, 70), (509, 5, 65), (512, 3, 64)])
def test_fp32_wide_summed_normals(gb, orc, d, steps, paths):
    w, pays = _case(d, 4, paths, steps)
    got = gb.price(gbm_model(w), cfg_of(w), pays)
    ref = oracle_gbm(orc, w, paths, pays)
    for i in range(2):
        m, se = orc.mean_se(ref[i])
        assert abs(got[i][0] - m) <= REL * max(abs(m), 1e-3 * se), (d, i, got[i], m)
        assert abs(got[i][1] - se) <= 1e-3 * se


@pytest.mark.parametrize("d,steps", [(2, 1), (3, 2), (5, 6), (18, 3), (31, 5), (64, 4)])
def test_fp32_basket_greeks_summed_normals(gb, orc, d, steps):
    w, pays = _case(d, 2, 700, steps)
    pr, g = gb.greeks(gbm_model(w), cfg_of(w), pays[:1])
    ref = orc.gbm_greeks(w["s0"], w["sigma"], w["r"], w["T"], steps, w["paths"], pays[:1], corr=w["corr"],
                         weights=w["weights"])[0]
    scale = np.max(np.abs(ref.mean(axis=1)[:d]))
    for k in range(2 * d + 1):
        m = ref[k].mean()
        assert abs(g[0, k, 0] - m) <= 2e-5 * max(abs(m), scale, np.mean(np.abs(ref[k]))), (d, k, g[0, k, 0], m)
