"""Nested revaluation of a slice of the scenarios: the bits of the same
scenarios in the whole run, whatever number of CTAs each run gives a
(scenario, underlying).  The runs lie on both sides of the count of pairs from
which the paths are no longer cut, with whole and ragged groups of paths."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_under,inner,base", [(4, 257, 1024), (4, 1024, 1025), (4, 1025, 5000), (4, 3001, 2048),
                                                (16, 2500, 70000)])
def test_shards_have_the_bits_of_the_whole_run(n_under, inner, base):
    import paper_1906_02818_gb300 as gb
    pf = workloads.risk_portfolio(n_under=n_under, per_under=8, seed=7)
    pf["maturity"] = np.resize(np.array([2, 3, 5, 6, 7, 12, 13, 63]) / 252.0, pf["maturity"].shape)
    n = 1024 if n_under == 4 else 256  # 4096 pairs
    kw = dict(inner_paths=inner, base_paths=base, seed=9, want_pnl=True)
    whole = gb.risk(pf, n_scen=n, **kw)
    at = 0
    for m in (1, 2, 7, 60, n // 4, n - 70 - n // 4):
        part = gb.risk(pf, n_scen=m, scen_offset=at, **kw)
        assert part["base_value"] == whole["base_value"]
        assert np.array_equal(part["pnl"], whole["pnl"][at:at + m]), (m, np.max(np.abs(part["pnl"] - whole["pnl"][at:at + m])))
        at += m
    assert at == n
