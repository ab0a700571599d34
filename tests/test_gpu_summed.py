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


@pytest.mark.parametrize("d,steps,paths", [(4, 3, 50000), (5, 6, 80001), (24, 2, 60000), (30, 3, 90000), (56, 2, 70000),
                                           (63, 1, 100001), (64, 2, 33000)])
def test_fp32_basket_greeks_many_paths(gb, d, steps, paths):
    """One and two paths per thread, whole and ragged last rounds: the sums over
    all paths are those of runs of at most 8192 of them (one path per thread)."""
    w, pays = _case(d, 2, paths, steps)
    pr, g = gb.greeks(gbm_model(w), cfg_of(w), pays[:1])
    total = np.zeros(2 * d + 2)
    for lo in range(0, paths, 8192):
        n = min(8192, paths - lo)
        p1, g1 = gb.greeks(gbm_model(w), cfg_of(dict(w, paths=n), path_offset=lo), pays[:1])
        total += n * np.concatenate([[p1[0][0]], np.asarray(g1)[0, :, 0]])
    got = np.concatenate([[pr[0][0]], np.asarray(g)[0, :, 0]])
    # the same FP32 terms in FP64 sums, rounded once per block of paths to FP32
    assert np.max(np.abs(got - total / paths)) <= 1e-6 * np.max(np.abs(got)), (d, got - total / paths)


@pytest.mark.parametrize("d,steps,paths", [(2, 1, 130), (3, 5, 129), (5, 3, 257), (7, 6, 128), (10, 4, 500),
                                           (18, 7, 131), (33, 2, 129), (47, 9, 127), (57, 5, 130), (63, 4, 200),
                                           (64, 3, 129)])
def test_fp32_basket_terminal_and_watched(gb, orc, d, steps, paths):
    """d <= 64: European payoffs (one contraction of the summed normals) and
    payoffs on the path (steps that start inside a Philox block)."""
    w, pays = _case(d, 2, paths, steps)
    b0 = pays[0]["strike"]
    for group in (pays, [dict(kind="asian_call", strike=b0), pays[1]]):
        got = gb.price(gbm_model(w), cfg_of(w), group)
        ref = oracle_gbm(orc, w, paths, group)
        for i in range(2):
            m, se = orc.mean_se(ref[i])
            assert abs(got[i][0] - m) <= REL * max(abs(m), 1e-3 * se), (d, group[i], got[i], m)
            assert abs(got[i][1] - se) <= 1e-3 * se


@pytest.mark.parametrize("d,steps,paths", [(5, 5, 80000), (30, 3, 90000), (50, 6, 100003), (56, 2, 70000), (40, 4, 130000)])
def test_fp32_basket_two_paths_per_thread(gb, orc, d, steps, paths):
    """Runs large enough for two paths per thread, with a ragged last round:
    the Asian price equals the FP64 oracle's on the same paths."""
    w, pays = _case(d, 2, paths, steps)
    group = [dict(kind="asian_call", strike=pays[0]["strike"])]
    got = gb.price(gbm_model(w), cfg_of(w), group)
    m, se = orc.mean_se(oracle_gbm(orc, w, paths, group)[0])
    assert abs(got[0][0] - m) <= REL * abs(m), (got, m)
    assert abs(got[0][1] - se) <= 1e-3 * se


@pytest.mark.parametrize("steps", [1, 2, 3, 4, 5, 6, 7])
def test_gbm1d_last_block(gb, orc, steps):
    """Path lengths around one Philox block: European (summed) and watched payoffs."""
    pays = [dict(kind="call", strike=100.0), dict(kind="asian_put", strike=101.0)]
    for group in (pays[:1], pays):
        got = gb.price(dict(kind="gbm", s0=[100.0], sigma=[0.3], r=0.02), dict(steps=steps, T=0.5, paths=777), group)
        ref = orc.gbm_payoffs(100.0, 0.3, 0.02, 0.5, steps, 777, group, seed=42)
        for i in range(len(group)):
            m, se = orc.mean_se(ref[i])
            assert abs(got[i][0] - m) <= REL * abs(m), (steps, i, got[i], m)


@pytest.mark.parametrize("steps", [1, 2, 7, 8, 9, 16, 23])
def test_heston_adjoint_strides_agree(gb, steps):
    """The register kernel (the default stride) and the general one run the
    same operations on the same states: the Greeks differ by the summation at most."""
    model = dict(kind="heston", s0=100.0, v0=0.04, r=0.05, kappa=2.0, theta=0.04, xi=0.5, rho=-0.7)
    pays = [dict(kind="call", strike=95.0), dict(kind="asian_call", strike=100.0), dict(kind="put", strike=105.0)]
    cfg = dict(steps=steps, T=0.5, paths=3001)
    p0, g0 = gb.greeks(model, cfg, pays)
    for k in (1, 8, 32, 64):
        p1, g1 = gb.greeks(model, dict(cfg, ckpt_every=k), pays)
        assert np.allclose(np.array(p0), np.array(p1), rtol=1e-6, atol=0)
        assert np.allclose(g0[..., 0], g1[..., 0], rtol=1e-5, atol=1e-5 * np.max(np.abs(g0[..., 0]), axis=1, keepdims=True))


@pytest.mark.parametrize("n_scen,inner", [(1, 700), (3, 256), (40, 300), (700, 33)])
def test_nested_slices(gb, n_scen, inner):
    """Few scenarios: the inner paths of a (scenario, underlying) are cut over
    several CTAs; many: not.  The PnL of a scenario does not depend on it."""
    import workloads
    pf = workloads.risk_portfolio(2, 16)
    pf["maturity"] = np.resize(np.array([2, 3, 5, 6, 7, 12, 13, 63]) / 252.0, pf["maturity"].shape)
    kw = dict(inner_paths=inner, base_paths=5000, seed=9, want_pnl=True)
    alone = gb.risk(pf, n_scen=n_scen, **kw)["pnl"]
    wide = gb.risk(pf, n_scen=1500, **kw)["pnl"][:n_scen]
    scale = np.abs(pf["strike"]).sum() * 0.1
    assert np.max(np.abs(alone - wide)) <= 2e-6 * scale, np.max(np.abs(alone - wide))


@pytest.mark.parametrize("d,steps,paths", [(5, 5, 70000), (16, 3, 100003), (24, 3, 130000), (30, 3, 100003), (40, 4, 70000),
                                           (50, 3, 100003), (56, 2, 100003), (48, 2, 160001)])
def test_fp32_euler_basket_paths_per_thread(gb, orc, d, steps, paths):
    """The Euler scheme, whose rule for two paths per thread is its own, on both
    sides of that rule: prices equal the FP64 oracle's on the same paths."""
    w, pays = _case(d, 2, paths, steps)
    for group in ([pays[0]], [dict(kind="asian_call", strike=pays[0]["strike"])]):
        got = gb.price(gbm_model(w), cfg_of(w, scheme="euler"), group)
        m, se = orc.mean_se(oracle_gbm(orc, w, paths, group, scheme="euler")[0])
        assert abs(got[0][0] - m) <= REL * abs(m), (d, group, got, m)
        assert abs(got[0][1] - se) <= 1e-3 * se


@pytest.mark.parametrize("d,steps,paths", [(17, 5, 3000), (17, 6, 3000), (40, 2, 20000), (48, 6, 9000), (48, 6, 9800),
                                           (57, 20, 31000), (64, 30, 30000)])
def test_fp32_basket_greeks_either_kernel(gb, orc, d, steps, paths):
    """Both sides of the rule that sends short or small runs to the
    large-basket kernel, against the FP64 oracle on the same paths.  One path
    whose basket value lies within rounding of the strike may fall on its other
    side: its whole term is allowed for."""
    w, pays = _case(d, 2, paths, steps)
    pr, g = gb.greeks(gbm_model(w), cfg_of(w), pays[:1])
    ref = orc.gbm_greeks(w["s0"], w["sigma"], w["r"], w["T"], steps, paths, pays[:1], corr=w["corr"], weights=w["weights"])[0]
    scale = np.max(np.abs(ref.mean(axis=1)[:d]))
    for k in range(2 * d + 1):
        m = ref[k].mean()
        tol = 2e-5 * max(abs(m), scale, np.mean(np.abs(ref[k]))) + np.max(np.abs(ref[k])) / paths
        assert abs(g[0, k, 0] - m) <= tol, (d, k, g[0, k, 0], m, tol)
