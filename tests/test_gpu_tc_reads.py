"""Reduced-precision baskets whose steps start inside a Philox block: every
residue of d mod 4, widths around the MMA's K and the 64 columns of a tile,
ragged tiles, against the quantised emulation."""
import pytest

from gpu_util import REL, cfg_of, gbm_model
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
