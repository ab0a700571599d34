"""Paths of more than 2^32 Philox blocks are read with 64-bit block indices, by
code of its own in every basket kernel.  No run in reach of a test is that long,
so the debug build takes those readers for every run when GBMC_DEBUG_WIDE=1 is
set: the results are those of the 32-bit readers, to the bit where both add the
same terms in the same order, else to the rounding of the FP32 sums."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys
import numpy as np
import paper_1906_02818_gb300 as gb
import workloads

def model(d):
    s0, sg, corr = workloads.basket_market(d, 3, seed=13)
    return dict(kind="gbm", s0=s0, sigma=sg, corr=corr, weights=np.full(d, 1.0 / d), r=0.05), float(np.mean(s0))

out = {}
for d, steps, paths in ((2, 1, 130), (3, 5, 200), (5, 6, 257), (13, 7, 129), (27, 4, 300), (30, 3, 131), (63, 4, 200), (64, 3, 300)):
    m, b = model(d)
    pays = [dict(kind="call", strike=b), dict(kind="uo_call", strike=b, barrier=1.3 * b), dict(kind="asian_put", strike=b)]
    for prec in ("fp32", "bf16", "fp16", "fp8"):
        for scheme in ("log_euler", "euler"):
            for name, group in (("terminal", pays[:1]), ("watched", pays)):
                cfg = dict(steps=steps, T=1.0, paths=paths, seed=7, precision=prec, scheme=scheme)
                out[f"price {prec} {scheme} {name} {d}"] = np.array(gb.price(m, cfg, group)).ravel().tolist()
    cfg = dict(steps=steps, T=1.0, paths=paths, seed=7)
    for kind in ("call", "asian_call"):
        r = gb.corr_greeks(m, cfg, dict(kind=kind, strike=b))
        out[f"corr {kind} {d}"] = np.concatenate([np.asarray(x, dtype=np.float64).ravel() for x in r]).tolist()
    p, g = gb.greeks(m, cfg, pays[:1])
    out[f"greeks {d}"] = np.concatenate([np.array(p).ravel(), g.ravel()]).tolist()
for d, steps, paths in ((65, 3, 130), (100, 5, 129), (130, 2, 64), (213, 3, 200), (512, 2, 65)):
    m, b = model(d)
    for prec in ("fp32", "bf16", "fp16", "fp8"):
        cfg = dict(steps=steps, T=1.0, paths=paths, seed=7, precision=prec)
        out[f"big {prec} {d}"] = np.array(gb.price(m, cfg, [dict(kind="call", strike=b)])).ravel().tolist()
        p, g = gb.greeks(m, cfg, [dict(kind="call", strike=b)])
        out[f"biggreeks {prec} {d}"] = np.concatenate([np.array(p).ravel(), g.ravel()]).tolist()
    r = gb.corr_greeks(m, dict(steps=steps, T=1.0, paths=paths, seed=7), dict(kind="call", strike=b))
    out[f"corr call {d}"] = np.concatenate([np.asarray(x, dtype=np.float64).ravel() for x in r]).tolist()
json.dump(out, open(sys.argv[1], "w"))
"""


def _run(lib, path, wide):
    env = dict(os.environ, GBMC_LIBRARY=lib, GBMC_DEBUG_WIDE="1" if wide else "0", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD, str(path)], cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, (r.stdout + r.stderr)[-3000:]
    return json.load(open(path))


def test_wide_readers_give_the_results_of_the_32_bit_ones(tmp_path):
    from paper_1906_02818_gb300 import build
    lib = build.build(debug=True)
    narrow, wide = _run(lib, tmp_path / "n.json", False), _run(lib, tmp_path / "w.json", True)
    assert list(narrow) == list(wide)
    for name, a in narrow.items():
        a, b = np.array(a), np.array(wide[name])
        # FP32 baskets up to 64 assets take another width (and Greeks another kernel): the sums' order differs; the
        # kernels of larger baskets add their warps' sums with atomics, in an order that differs between two runs of
        # the same kernel.  A path's value and its sum over at most 300 paths round at 2^-24 each; a step adds at
        # most 64 products in another order: 1e-5 of the largest value covers them.
        if name.startswith(("price fp32", "greeks", "big")):
            assert np.allclose(b, a, rtol=1e-5, atol=1e-5 * np.max(np.abs(a))), (name, np.max(np.abs(a - b)))
        else:
            assert np.array_equal(a, b, equal_nan=True), (name, np.max(np.abs(a - b)))
