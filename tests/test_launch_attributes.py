"""Shared-memory attributes of the kernels, and calls from several threads.

cudaFuncSetAttribute changes the process's state, and a launch that asks for
more dynamic shared memory than the attribute allows fails.  Host threads may be
between the setting and the launch at once, so a function's attribute has to be
the same in every call: no setting may take its size from the call."""
import glob
import os
import re
import threading

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_02818_gb300", "csrc")
# sizes that go with the call's assets, factors, payoffs or width
VARYING = re.compile(r"greeks_slots|greeks_smem|factor_smem_bytes|corr_adjoint_smem\(a\.d\)|a\.W|n_payoff|a\.pay\.n")


def _settings():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(f).read()
        for m in re.finditer(r"cudaFuncSetAttribute\(", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            size = text[m.end():i - 1].split("MaxDynamicSharedMemorySize,")[1]
            name = re.fullmatch(r"\s*(?:static_cast<int>\()?(\w+)\)?\s*", size)
            if name:  # a variable: its definition above
                size += "".join(re.findall(r"\b" + name[1] + r" = ([^;]*);", text[max(0, m.start() - 600):m.start()])[-1:])
            yield os.path.basename(f), size


def test_every_attribute_is_the_functions_own():
    seen = list(_settings())
    assert len(seen) >= 6
    for f, size in seen:
        assert not VARYING.search(size), (f, size)


@pytest.mark.gpu
def test_threads_get_the_results_of_one():
    """Calls of several sizes at a time on the kernels whose shared memory goes
    with the call, and on the price call's host result blocks."""
    import torch
    import paper_1906_02818_gb300 as gb
    import workloads

    def model(d):
        s0, sg, corr = workloads.basket_market(d, 4)
        return dict(kind="gbm", s0=s0, sigma=sg, corr=corr, r=0.05)

    def basket(d, paths):
        m = model(d)
        return lambda s: gb.greeks(m, dict(steps=1, T=1.0, paths=paths), [dict(kind="call", strike=100.0)], stream=s)

    def corr(d):
        m = model(d)
        return lambda s: gb.corr_greeks(m, dict(steps=1, T=1.0, paths=64), dict(kind="call", strike=100.0), stream=s)

    def heston(n):
        m = dict(kind="heston", s0=100.0, v0=0.04, r=0.05, kappa=2.0, theta=0.04, xi=0.5, rho=-0.7)
        return lambda s: gb.greeks(m, dict(steps=2, T=1.0, paths=64), [dict(kind="call", strike=90.0 + i) for i in range(n)],
                                   stream=s)

    def price(paths):
        return lambda s: gb.price(dict(kind="gbm", s0=[100.0], sigma=[0.2], r=0.05), dict(steps=4, T=1.0, paths=paths),
                                  [dict(kind="call", strike=100.0), dict(kind="put", strike=90.0)], stream=s)

    def flat(r):
        if isinstance(r, (tuple, list)):
            return np.concatenate([flat(x) for x in r])
        return np.asarray(r, dtype=np.float64).ravel()

    jobs = [basket(63, 1 << 17), basket(57, 64), corr(64), corr(50), heston(1), heston(20), price(500), price(70000)]
    main = torch.cuda.current_stream()
    want = [flat(j(main)) for j in jobs]
    wrong = []

    def work(k):
        s = torch.cuda.Stream()
        for _ in range(150):
            try:
                if not np.array_equal(flat(jobs[k](s)), want[k], equal_nan=True):
                    wrong.append((k, "values"))
            except Exception as e:  # noqa: BLE001
                wrong.append((k, str(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, (len(wrong), wrong[:3])
