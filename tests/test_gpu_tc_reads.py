"""Reduced-precision baskets whose steps start inside a Philox block: every
residue of d mod 4, widths around the MMA's K, the 64 columns of a panel and
the 128 rows of a factor block, ragged tiles, against the quantised emulation."""
import numpy as np
import pytest

from gpu_util import REL, cfg_of, gbm_model
from test_gpu_big import _case as big_case
from test_gpu_tc import _case, band, emulate, flip_bound, payoffs_from_U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import torch
    assert torch.cuda.is_available()
    import paper_1906_02818_gb300 as gb
    return gb


@pytest.mark.parametrize("prec", ["bf16", "fp16", "fp8"])
@pytest.mark.parametrize("d,steps,scheme", [(2, 1, "log_euler"), (3, 5, "log_euler"), (5, 2, "log_euler"), (16, 3, "log_euler"),
                                            (17, 6, "log_euler"), (31, 4, "euler"), (33, 7, "log_euler"),
                                            (50, 3, "euler"), (63, 5, "log_euler")])
def test_tc_any_width(gb, orc, prec, d, steps, scheme):
    w, pays = _case(d, 2, 261, steps)
    got = gb.price(gbm_model(w), cfg_of(w, precision=prec, scheme=scheme), pays)
    euro = gb.price(gbm_model(w), cfg_of(w, precision=prec, scheme=scheme), pays[:2])
    U, aux = emulate(orc, w, prec, w["paths"], steps, scheme, detail=True)
    want = payoffs_from_U(U, pays, w["r"], w["T"])
    bm = band(U, pays, want)
    fb = flip_bound(aux, U, pays, w["r"], w["T"])
    for i, p in enumerate(pays):
        m = want[i].mean()
        tol = REL * max(abs(m), 1e-6) + bm[i] + fb[i]
        assert abs(got[i][0] - m) <= tol, (prec, d, scheme, p, got[i][0], m, tol)
        if i < 2:
            assert abs(euro[i][0] - m) <= tol, (prec, d, scheme, p, euro[i][0], m, tol)


@pytest.mark.parametrize("prec", ["bf16", "fp16", "fp8"])
@pytest.mark.parametrize("d,steps,paths", [(65, 1, 129), (66, 3, 127), (67, 5, 60), (68, 2, 130), (127, 7, 100),
                                           (130, 4, 128), (193, 2, 90), (257, 6, 50), (510, 5, 40), (511, 3, 40)])
def test_tc_big_any_width(gb, orc, prec, d, steps, paths):
    w, pays = big_case(d, 4, paths, steps)
    got = gb.price(gbm_model(w), cfg_of(w, precision=prec), pays)
    U, aux = emulate(orc, w, prec, paths, steps, fp8_fixed=True, detail=True)
    want = payoffs_from_U(U, pays, w["r"], w["T"])
    fb = flip_bound(aux, U, pays, w["r"], w["T"])
    for i in range(2):
        m = want[i].mean()
        assert abs(got[i][0] - m) <= 2 * REL * max(abs(m), 1e-6) + fb[i], (prec, d, i, got[i][0], m)


@pytest.mark.parametrize("prec,d,steps,paths", [("bf16", 65, 9, 40001), ("fp8", 130, 6, 20000), ("bf16", 258, 5, 39000),
                                                ("fp16", 323, 3, 20011), ("bf16", 511, 4, 58500), ("fp8", 512, 3, 41000)])
def test_tc_big_many_tiles(gb, prec, d, steps, paths):
    """Several tiles per CTA (the rings of panels and factor chunks wrap from one
    to the next), equal to runs of at most one tile per CTA: FP32 sums in another order."""
    w, pays = big_case(d, 4, paths, steps)
    got = gb.price(gbm_model(w), cfg_of(w, precision=prec), pays)
    total = np.zeros(2)
    for lo in range(0, paths, 8192):
        n = min(8192, paths - lo)
        part = gb.price(gbm_model(w), cfg_of(dict(w, paths=n), precision=prec, path_offset=lo), pays)
        total += n * np.array([p[0] for p in part])
    want = total / paths
    for i in range(2):
        assert abs(got[i][0] - want[i]) <= REL * abs(want[i]), (prec, d, i, got[i], want[i])
