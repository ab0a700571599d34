"""Performance cases of the Monte Carlo library: the calls a user's program makes, over the sizes it makes them at.

A case is a dict of plain values; "what" names its family:

  price    gb.price, or a gb.Plan executed again and again ("plan"): discounted prices and standard errors of a
           GBM asset (d = 1), a correlated GBM basket (2 <= d <= 64, path-dependent payoffs) or a large one (d > 64,
           European payoffs), in FP32 or with the reduced-precision contraction
  heston   prices and gradient of a book of European and Asian calls through gb.HestonPricer (model calibration)
  grad     price and gradient of a basket option in spot, volatility, rate and correlation through gb.BasketPricer
  labels   Monte Carlo training labels of the pricing network with their pathwise delta and vega
  train    loss and parameter gradient of one mini-batch of prices and Greeks (gb.Mlp.loss_grad_d)
  risk     VaR / CVaR of an option portfolio, revalued by the network or by nested Monte Carlo (gb.risk)

Everything comes from the seed.  `exact` repeats the same random stream (Philox4x32-10, Box-Muller) and the same
estimators in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1906_02818_gb300 as gb

RATE = 0.05


# ------------------------------------------------------------- the cases
def listed():
    return [
        # a desk's quote of one option sheet: launch and set-up latency
        dict(name="quote_1d", what="price", d=1, paths=4096, steps=64, precision="fp32",
             payoffs="call,asian_call,uo_call", plan=False),
        # one European call at a million paths
        dict(name="call_1d", what="price", d=1, paths=1 << 20, steps=64, precision="fp32", payoffs="call", plan=False),
        # the 64-name basket with a daily-monitored barrier, repriced through its plan
        dict(name="basket64_bf16", what="price", d=64, paths=1 << 18, steps=252, precision="bf16",
             payoffs="call,uo_call", plan=True),
        # a basket of no round size with averages and a lower barrier, in the default precision
        dict(name="basket50_fp32", what="price", d=50, paths=100003, steps=100, precision="fp32",
             payoffs="asian_call,put,do_put", plan=False),
        # an index-sized basket in reduced precision
        dict(name="basket512_bf16", what="price", d=512, paths=1 << 17, steps=252, precision="bf16", payoffs="call",
             plan=True),
        # the same index in the default precision
        dict(name="basket512_fp32", what="price", d=512, paths=1 << 16, steps=252, precision="fp32", payoffs="call",
             plan=False),
        # one calibration step of a Heston model: 18 options and the gradient of their weighted sum
        dict(name="heston_grad", what="heston", paths=1 << 22, steps=256, strikes=9),
        # a basket call's price with every first-order sensitivity, correlation included
        dict(name="basket64_grad", what="grad", d=64, paths=1 << 18, steps=252, payoff="call"),
        # labels of a batch of training points
        dict(name="labels", what="labels", points=4096, paths=1 << 13),
        # one mini-batch of the network's training on prices and Greeks
        dict(name="train_step", what="train", batch=4096, width=256, hidden=4, dirs=2, mode="tf32x3"),
        # the overnight VaR of a thousand options through the network
        dict(name="risk_network", what="risk", method="surrogate", scenarios=1 << 16, under=32, per_under=32,
             inner=0, precision="bf16"),
        # the nested revaluation that the network is checked against
        dict(name="risk_nested", what="risk", method="nested", scenarios=512, under=32, per_under=32, inner=1024,
             precision="fp32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["price1", "price", "price", "large", "large", "heston", "grad", "labels", "train", "network",
                       "nested"])
    if what == "price1":
        return dict(what="price", d=1, paths=_log(rng, 1000, 1 << 22), steps=_log(rng, 1, 365), precision="fp32",
                    payoffs=rng.choice(["call", "put,asian_put", "call,asian_call,uo_call", "ui_put", "do_call,put"]),
                    plan=rng.random() < 0.5)
    if what == "price":
        d, steps = rng.randint(2, 64), _log(rng, 4, 252)
        top = (1 << 18) * 252 * 64 // (d * steps)
        return dict(what="price", d=d, paths=_log(rng, 1000, min(top, 1 << 20)), steps=steps,
                    precision=rng.choice(["fp32", "fp32", "bf16", "bf16", "fp16", "fp8"]),
                    payoffs=rng.choice(["call", "call,put", "call,uo_call", "asian_call", "do_put,put"]),
                    plan=rng.random() < 0.5)
    if what == "large":
        d, steps, precision = rng.randint(65, 512), _log(rng, 4, 252), rng.choice(["fp32", "bf16", "fp16", "fp8"])
        top = (1 << 16) * 252 * 512 // (d * steps)
        return dict(what="price", d=d, paths=_log(rng, 1000, min(top, 1 << 19)), steps=steps, precision=precision,
                    payoffs=rng.choice(["call", "put", "call,put"]), plan=rng.random() < 0.5)
    if what == "heston":
        return dict(what="heston", paths=_log(rng, 4096, 1 << 21), steps=_log(rng, 12, 365), strikes=rng.randint(1, 9))
    if what == "grad":
        d, steps = _log(rng, 2, 160), _log(rng, 4, 252)
        top = (1 << 17) * 252 * 64 // (d * steps)
        return dict(what="grad", d=d, paths=_log(rng, 4096, min(top, 1 << 20)), steps=steps,
                    payoff=rng.choice(["call", "put"]))
    if what == "labels":
        return dict(what="labels", points=_log(rng, 64, 4096), paths=_log(rng, 256, 1 << 13))
    if what == "train":
        return dict(what="train", batch=_log(rng, 256, 8192), width=rng.choice([64, 128, 256]),
                    hidden=rng.randint(2, 5), dirs=rng.randint(0, 2), mode=rng.choice(["fp32", "tf32x3"]))
    under = rng.randint(4, 48)
    if what == "network":
        return dict(what="risk", method="surrogate", scenarios=_log(rng, 500, 1 << 14), under=under,
                    per_under=rng.randint(8, 32), inner=0, precision=rng.choice(["bf16", "bf16", "fp32"]))
    top = 512 * 32 * 1024 // under
    inner = _log(rng, 128, 4096)
    return dict(what="risk", method="nested", scenarios=_log(rng, 64, max(65, min(512, top // inner))), under=under,
                per_under=rng.randint(8, 32), inner=inner, precision="fp32")


# ------------------------------------------------- inputs, from the seed
def _market(d, seed):
    """Spots, volatilities, correlation (a few factors and a ridge) and weights of d names."""
    rng = np.random.default_rng(seed)
    s0, sigma = rng.uniform(50.0, 150.0, d), rng.uniform(0.1, 0.4, d)
    k = 16 if d > 64 else 4
    F = rng.standard_normal((d, k))
    C = F @ F.T / k + 0.05 * np.eye(d)
    s = 1.0 / np.sqrt(np.diag(C))
    corr = C * s[:, None] * s[None, :]
    corr = 0.5 * (corr + corr.T)
    np.fill_diagonal(corr, 1.0)
    return s0, sigma, corr, np.full(d, 1.0 / d)


def _price_inputs(case, seed):
    d = case["d"]
    s0, sigma, corr, w = _market(d, seed)
    b0 = float(w @ s0)
    payoffs = []
    for kind in case["payoffs"].split(","):
        p = dict(kind=kind, strike=b0 if kind.endswith("call") else 1.05 * b0)  # a put at the money forward
        if kind[:2] in ("uo", "ui"):
            p["barrier"] = 1.3 * b0
        if kind[:2] in ("do", "di"):
            p["barrier"] = 0.8 * b0
        payoffs.append(p)
    model = dict(kind="gbm", s0=s0, sigma=sigma, r=RATE, weights=w)
    if d > 1:
        model["corr"] = corr
    return model, dict(steps=case["steps"], T=1.0, paths=case["paths"], seed=seed, precision=case["precision"]), payoffs


def _heston_inputs(case, seed):
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1.0, 1.0, 7)
    p = np.array([100.0 + 5 * x[0], 0.04 + 0.01 * x[1], RATE + 0.01 * x[2], 2.0 + 0.3 * x[3], 0.04 + 0.01 * x[4],
                  0.5 + 0.1 * x[5], -0.7 + 0.1 * x[6]], dtype=np.float32)
    n = case["strikes"]
    strikes = [100.0 + 5.0 * (i - (n - 1) / 2) for i in range(n)]
    payoffs = [dict(kind=k, strike=s) for k in ("call", "asian_call") for s in strikes]
    weight = rng.uniform(0.2, 1.0, 2 * n).astype(np.float32)  # the residuals of a least-squares fit
    return p, dict(steps=case["steps"], T=1.0, paths=case["paths"], seed=seed), payoffs, weight


def _grad_inputs(case, seed):
    s0, sigma, corr, w = _market(case["d"], seed)
    payoff = dict(kind=case["payoff"], strike=(1.0 if case["payoff"] == "call" else 1.05) * float(w @ s0))
    f = [np.asarray(a, dtype=np.float32) for a in (s0, sigma, RATE, corr)]
    return f, dict(steps=case["steps"], T=1.0, paths=case["paths"], seed=seed), payoff, w


def _points(n, seed):
    """Points (S/K, sigma, tau, r, K/H) of the network's box; half of them without a barrier (K/H = 0)."""
    rng = np.random.default_rng(seed)
    x = np.empty((n, 5))
    x[:, 0] = rng.uniform(0.5, 1.6, n)
    x[:, 1] = rng.uniform(0.1, 0.4, n)
    x[:, 2] = rng.integers(1, 505, n) / 252.0
    x[:, 3] = rng.uniform(0.0, 0.08, n)
    x[:, 4] = np.where(rng.uniform(size=n) < 0.5, 0.0, rng.uniform(0.5, 0.9, n))
    return x.astype(np.float32)


SLOPE, SHIFT = np.array([0.55, 0.15, 1.0, 0.04, 0.45]), np.array([1.05, 0.25, 1.0, 0.04, 0.45])


def _net(width, hidden, seed):
    rng = np.random.default_rng(seed)
    sizes, parts = [5] + [width] * hidden + [1], []
    for a, b in zip(sizes[:-1], sizes[1:]):
        parts += [(rng.standard_normal((a, b)) / math.sqrt(a)).ravel(), 0.1 * rng.standard_normal(b)]
    return np.concatenate(parts).astype(np.float32), sizes


def _train_inputs(case, seed):
    n = case["batch"]
    p = _points(n, seed).astype(np.float64)
    net, sizes = _net(case["width"], case["hidden"], seed + 1)
    # Black-Scholes values and Greeks with the noise of a few thousand paths stand for the labels
    rng = np.random.default_rng(seed + 2)
    t = torch.from_numpy(p)
    sk, sg, tau, r = t[:, 0], t[:, 1], t[:, 2], t[:, 3]
    sd = sg * tau.sqrt()
    d1 = (sk.log() + (r + 0.5 * sg * sg) * tau) / sd
    N = lambda v: 0.5 * (1 + torch.erf(v / math.sqrt(2.0)))  # noqa: E731
    price = sk * N(d1) - torch.exp(-r * tau) * N(d1 - sd)
    delta, vega = N(d1), sk * tau.sqrt() * torch.exp(-0.5 * d1 * d1) / math.sqrt(2 * math.pi)
    g = np.stack([delta.numpy(), vega.numpy()], 1) + 5e-3 * rng.standard_normal((n, 2))
    g[p[:, 4] > 0] = np.nan  # a barrier point has no Greek label
    y = price.numpy() + 2e-3 * rng.standard_normal(n)
    x = (p - SHIFT) / SLOPE
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    return net, sizes, f32(x), f32(y), f32(g[:, :case["dirs"]])


DIRS, SCALES, WEIGHTS = (0, 1), (1 / 0.55, 1 / 0.15), (0.2, 0.05)


def _portfolio(case, seed):
    """Half European calls and puts, half daily up-and-out calls on every underlying; positions +-1."""
    u, per = case["under"], case["per_under"]
    s0, sigma, corr, _ = _market(u, seed)
    rng = np.random.default_rng(seed + 1)
    n = u * per
    under = np.repeat(np.arange(u), per)
    barrier = np.tile(np.arange(per) >= per // 2, u)
    kind = np.where(barrier, 4, rng.integers(0, 2, n)).astype(np.int32)
    K = np.where(barrier, rng.choice([0.8, 0.9, 1.0], n), rng.choice([0.8, 0.9, 1.0, 1.1, 1.2], n)) * s0[under]
    H = np.where(barrier, rng.uniform(1.2, 1.5, n) * s0[under], np.inf)
    return dict(s0=s0, sigma=sigma, corr=corr, r=RATE, mu=RATE, under=under.astype(np.int32), kind=kind, strike=K,
                barrier=H, maturity=rng.choice([63, 126, 252, 504], n) / 252.0, position=rng.choice([-1.0, 1.0], n),
                horizon=1.0 / 252, steps_per_year=252)


# --------------------------------------------------------------- a pass
def prepare(case, seed):
    what = case["what"]
    if what == "price":
        model, cfg, payoffs = _price_inputs(case, seed)
        plan = gb.Plan(model, cfg, payoffs) if case["plan"] else None
        return dict(what=what, model=model, cfg=cfg, payoffs=payoffs, plan=plan)
    if what == "heston":
        p, cfg, payoffs, weight = _heston_inputs(case, seed)
        return dict(what=what, params=torch.from_numpy(p).requires_grad_(), cfg=cfg, payoffs=payoffs,
                    weight=torch.from_numpy(weight))
    if what == "grad":
        f, cfg, payoff, w = _grad_inputs(case, seed)
        return dict(what=what, params=[torch.tensor(a).requires_grad_() for a in f], cfg=cfg, payoff=payoff, weights=w)
    if what == "labels":
        return dict(what=what, points=torch.from_numpy(_points(case["points"], seed)).cuda(), paths=case["paths"],
                    seed=seed)
    if what == "train":
        net, _, x, y, g = _train_inputs(case, seed)
        mlp = gb.Mlp(5, case["width"], case["hidden"], net)
        mlp.set_train_mode(case["mode"])
        k = case["dirs"]
        return dict(what=what, mlp=mlp, x=torch.from_numpy(x).cuda(), y=torch.from_numpy(y).cuda(),
                    g=torch.from_numpy(g).cuda(), loss=(DIRS[:k], SCALES[:k], WEIGHTS[:k]))
    net = gb.Mlp(5, 256, 4, _net(256, 4, seed + 1)[0]) if case["method"] == "surrogate" else None
    return dict(what=what, portfolio=_portfolio(case, seed), net=net, case=case, seed=seed)


def run(s):
    what = s["what"]
    if what == "price":
        if s["plan"] is not None:
            return s["plan"].execute().tolist()  # the program reads its prices
        return gb.price(s["model"], s["cfg"], s["payoffs"])
    if what == "heston":
        prices = gb.HestonPricer.apply(s["params"], s["cfg"], s["payoffs"])
        return [prices.detach(), torch.autograd.grad(prices, s["params"], s["weight"])[0]]
    if what == "grad":
        price = gb.BasketPricer.apply(*s["params"], s["cfg"], s["payoff"], s["weights"])
        return [price.detach(), *torch.autograd.grad(price, s["params"])]
    if what == "labels":
        return list(gb.surrogate_label_greeks(s["points"], s["paths"], seed=s["seed"]))
    if what == "train":
        return s["mlp"].loss_grad_d(s["x"], s["y"], s["g"], *s["loss"])
    c = s["case"]
    return gb.risk(s["portfolio"], n_scen=c["scenarios"], method=c["method"], inner_paths=max(c["inner"], 1),
                   surrogate=s["net"], surrogate_precision=c["precision"], seed=s["seed"])


# ------------------------------------------- what a pass cannot do without
NORMAL = 20  # operations of one normal: a quarter of ten Philox rounds (four operations each), half a Box-Muller pair


def work(case):
    """Every normal drawn once and added to its asset's running sum; the contraction of a path once per monitored date,
    or once at maturity where no payoff looks at the path in between."""
    what = case["what"]
    if what == "price":
        d, n, m = case["d"], case["paths"], case["steps"]
        dates = 1 if set(case["payoffs"].split(",")) <= {"call", "put"} else m
        return dict(bytes=8 * d * (d + 4), flops=n * (m * d * (NORMAL + 1) + dates * (d * (d + 1) + 3 * d)))
    if what == "heston":
        n, m = case["paths"], case["steps"]
        return dict(bytes=200, flops=n * m * (3 * (2 * NORMAL) + 20 + 60))  # priced, run forward, run back
    if what == "grad":
        d, n, m = case["d"], case["paths"], case["steps"]
        return dict(bytes=8 * d * (2 * d + 8), flops=n * (2 * m * d * (NORMAL + 1) + 2 * d * (d + 1) + 2 * d * d))
    if what == "labels":
        n, m = case["points"] * case["paths"], 252.5
        return dict(bytes=case["points"] * 32, flops=n * m * (NORMAL + 3))
    if what == "train":
        w, h, n = case["width"], case["hidden"], case["batch"]
        rows = n * (1 + case["dirs"])
        params = 5 * w + (h - 1) * w * w + w
        return dict(bytes=4 * (2 * params + n * (6 + case["dirs"])), flops=6.0 * rows * params)
    n, u, o = case["scenarios"], case["under"], case["under"] * case["per_under"]
    if case["method"] == "surrogate":
        return dict(bytes=4 * (6 * 256 + 3 * 65536) + 40 * o, flops=2.0 * n * o * (6 * 256 + 3 * 65536))
    return dict(bytes=40 * o, flops=u * (n * case["inner"] + 65536.0) * 504 * (NORMAL + 3))


# ----------------------------------------------------- the same, in 64 bits
M32 = 0xFFFFFFFF


def _words(q, n, seed):
    """Philox4x32-10 of counters (q, n) (int64 tensors of one shape): four int64 tensors of 32-bit words."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    x, y, z, w = q & M32, (q >> 32) & M32, n & M32, (n >> 32) & M32
    for _ in range(10):
        p0, p1 = x * 0xD2511F53, z * 0xCD9E8D57
        x, z = (p1 >> 32).bitwise_and_(M32).bitwise_xor_(y).bitwise_xor_(k0), \
            (p0 >> 32).bitwise_and_(M32).bitwise_xor_(w).bitwise_xor_(k1)
        y, w = p1.bitwise_and_(M32), p0.bitwise_and_(M32)
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return x, y, z, w


def _normals(q0, blocks, n, seed):
    """Normals 4 q0 .. 4 (q0 + blocks) - 1 of the streams n [P]: [4 blocks, P], float64."""
    q = torch.arange(q0, q0 + blocks, dtype=torch.int64, device=n.device)[:, None].expand(blocks, n.numel())
    words = _words(q.contiguous(), n[None, :].expand(blocks, -1).contiguous(), seed)
    u = [((x >> 9).double() + 0.5) * 2.0 ** -23 for x in words]
    out = torch.empty((blocks, 4, n.numel()), dtype=torch.float64, device=n.device)
    for i in (0, 2):
        r, th = (u[i].log() * -2.0).sqrt_(), u[i + 1] * (2 * math.pi)
        out[:, i], out[:, i + 1] = r * th.cos(), r * th.sin()
    return out.view(4 * blocks, -1)


def _steps(n, d, steps, seed):
    """Yields the normals [d, P] of every step of the streams n."""
    per = max(1, (1 << 20) // max(1, n.numel() * max(1, d // 4)))  # steps drawn at a time
    for i in range(0, steps, per):
        a, b = i * d, min(steps, i + per) * d
        z = _normals(a // 4, (b + 3) // 4 - a // 4, n, seed)[a - a // 4 * 4:]
        for j in range((b - a) // d):
            yield z[j * d:(j + 1) * d]


def _mean_se(f, disc):
    n = f.numel()
    m = f.mean()
    var = ((f * f).mean() - m * m).clamp_min(0.0)
    return disc * float(m), disc * math.sqrt(float(var) / (n - 1))


def _chunks(paths, d):
    size = max(1024, (1 << 22) // d)
    for i in range(0, paths, size):
        yield torch.arange(i, min(paths, i + size), dtype=torch.int64, device="cuda")


def _exact_price(case, seed):
    model, cfg, payoffs = _price_inputs(case, seed)
    d, m = case["d"], cfg["steps"]
    dt = cfg["T"] / m
    T = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    s0, sg, w = T(model["s0"]), T(model["sigma"]), T(model["weights"])
    L = T(np.linalg.cholesky(model["corr"]) if d > 1 else np.ones((1, 1))) * (sg * math.sqrt(dt))[:, None]
    drift, ws0 = (RATE - 0.5 * sg * sg) * dt, w * s0
    terminal = all(p["kind"] in ("call", "put") for p in payoffs)
    parts = []
    for n in _chunks(case["paths"], d):
        x = torch.zeros((d, n.numel()), dtype=torch.float64, device="cuda")
        if terminal:
            for z in _steps(n, d, m, cfg["seed"]):
                x += z
            U = ws0 @ torch.exp(L @ x + m * drift[:, None])
            tot, hi, lo = U, U, U
        else:
            tot = hi = lo = None
            for z in _steps(n, d, m, cfg["seed"]):
                x += L @ z + drift[:, None]
                U = ws0 @ torch.exp(x)
                tot, hi, lo = (U, U, U) if tot is None else (tot + U, torch.maximum(hi, U), torch.minimum(lo, U))
        f = []
        for p in payoffs:
            kind, K, H = p["kind"], p["strike"], p.get("barrier")
            u = tot / m if kind.startswith("asian") else U
            v = (u - K if kind.endswith("call") else K - u).clamp_min(0.0)
            if H is not None:
                hit = hi >= H if kind[0] == "u" else lo <= H
                v = torch.where(hit if kind[1] == "i" else ~hit, v, torch.zeros_like(v))
            f.append(v)
        parts.append(torch.stack(f))
    f = torch.cat(parts, 1)
    return [_mean_se(v, math.exp(-RATE * cfg["T"])) for v in f]


def _exact_heston(case, seed):
    p, cfg, payoffs, weight = _heston_inputs(case, seed)
    s0, v0, r, kappa, theta, xi, rho = (float(a) for a in p)
    m = cfg["steps"]
    dt, rhoc = 1.0 / m, math.sqrt(1 - rho * rho)
    disc = math.exp(-r)
    price, grad = torch.zeros(len(payoffs), dtype=torch.float64), torch.zeros(7, dtype=torch.float64)
    size = 1 << 19
    for i in range(0, case["paths"], size):
        n = torch.arange(i, min(case["paths"], i + size), dtype=torch.int64, device="cuda")
        P = n.numel()
        x, v = torch.zeros(P, dtype=torch.float64, device="cuda"), torch.full((P,), v0, dtype=torch.float64, device="cuda")
        dx, dv = (torch.zeros((6, P), dtype=torch.float64, device="cuda") for _ in range(2))  # v0 r kappa theta xi rho
        dv[0] = 1.0
        tot, dtot = torch.zeros_like(x), torch.zeros_like(dx)
        for z in _steps(n, 2, m, cfg["seed"]):
            z1, z2 = z[0], z[1]
            vp = v.clamp_min(0.0)
            sq = (vp * dt).sqrt()
            c = rho * z1 + rhoc * z2
            dvp = dv * (v > 0)
            dsq = dvp * torch.where(v > 0, 0.5 * dt / sq, torch.zeros_like(v))
            dx = dx + dsq * c - 0.5 * dt * dvp
            dx[1] += dt
            dx[5] += sq * (z1 - rho / rhoc * z2)
            dv = dv + xi * dsq * z1 - kappa * dt * dvp
            dv[2] += (theta - vp) * dt
            dv[3] += kappa * dt
            dv[4] += sq * z1
            x = x + sq * c + (r - 0.5 * vp) * dt
            v = v + xi * sq * z1 + kappa * (theta - vp) * dt
            S = s0 * torch.exp(x)
            tot += S
            dtot += S * dx
        for k, q in enumerate(payoffs):
            u, du = (S, S * dx) if q["kind"] == "call" else (tot / m, dtot / m)
            f, on = (u - q["strike"]).clamp_min(0.0), (u > q["strike"]).double()
            price[k] += float(f.sum())
            g = [float((on * u).sum()) / s0] + [float(t) for t in (du * on).sum(1)]
            g[2] -= float(f.sum())
            grad += float(weight[k]) * torch.tensor(g, dtype=torch.float64)
    return [price * disc / case["paths"], grad * disc / case["paths"]]


def _exact_grad(case, seed):
    (s0, sg, r, corr), cfg, payoff, w = _grad_inputs(case, seed)
    d, m, T = case["d"], cfg["steps"], cfg["T"]
    par = [torch.tensor(a, dtype=torch.float64, device="cuda").requires_grad_() for a in (s0, sg, r, corr)]
    w = torch.as_tensor(w, dtype=torch.float64, device="cuda")
    sign = 1.0 if payoff["kind"] == "call" else -1.0
    total, grads = 0.0, [torch.zeros_like(p) for p in par]
    for n in _chunks(case["paths"], d):
        W = torch.zeros((d, n.numel()), dtype=torch.float64, device="cuda")
        for z in _steps(n, d, m, cfg["seed"]):
            W += z
        a, b, c, rho = par
        x = (c - 0.5 * b * b)[:, None] * T + math.sqrt(T / m) * b[:, None] * (torch.linalg.cholesky(rho) @ W)
        f = (sign * ((w * a) @ torch.exp(x) - payoff["strike"])).clamp_min(0.0).sum() * torch.exp(-c * T) / case["paths"]
        for t, g in zip(grads, torch.autograd.grad(f, par)):
            t += g
        total += float(f.detach())
    grads[3].fill_diagonal_(0.0)
    return [torch.tensor(total, dtype=torch.float64), *grads]


def _exact_labels(case, seed):
    pts, paths = _points(case["points"], seed).astype(np.float64), case["paths"]
    lab, dlab = np.empty(len(pts)), np.full((len(pts), 2), np.nan)
    per = max(1, (1 << 16) // paths)
    days = np.maximum(1, np.rint(pts[:, 2] * 252)).astype(int)
    order = np.argsort(days, kind="stable")
    for i in range(0, len(pts), per):
        at = order[i:i + per]
        t = torch.from_numpy(pts[at]).cuda().repeat_interleave(paths, 0)
        sk, sg, tau, r, kh = t.unbind(1)
        m = torch.from_numpy(days[at]).cuda().repeat_interleave(paths)
        n = (4 << 56) | (torch.from_numpy(at).cuda().repeat_interleave(paths) << 16) | torch.arange(
            paths, device="cuda").repeat(len(at))
        dt = tau / m
        top = int(days[at].max())
        y, zs = torch.zeros_like(sk), torch.zeros_like(sk)
        alive = ~((kh > 0) & (sk * kh >= 1))
        drift, vol = (r - 0.5 * sg * sg) * dt, sg * dt.sqrt()
        logh = torch.where(kh > 0, -torch.log(sk * kh.clamp_min(1e-30)), torch.full_like(kh, math.inf))
        ragged = bool((m != top).any())
        for q in range(0, top, 64):
            z = _normals(q // 4, (min(64, top - q) + 3) // 4, n, seed)[:top - q]
            if ragged:
                z = torch.where(torch.arange(q, q + len(z), device="cuda")[:, None] < m, z, torch.zeros_like(z))
            path = y + torch.cumsum(vol * z, 0)
            k = torch.arange(q + 1, q + len(z) + 1, dtype=torch.float64, device="cuda")[:, None]
            k = torch.minimum(k, m) if ragged else k
            alive &= ((path + drift * k) < logh).all(0)
            y, zs = path[-1], zs + z.sum(0)
        g = torch.exp(y + drift * m)
        ST, on = sk * g, (sk * g > 1).double()
        disc = np.exp(-pts[at, 3] * pts[at, 2])
        mean = lambda v: v.view(len(at), paths).mean(1).cpu().numpy()  # noqa: E731
        lab[at] = disc * mean(torch.where(alive, (ST - 1).clamp_min(0.0), torch.zeros_like(ST)))
        both = np.stack([disc * mean(on * g), disc * mean(on * ST * (dt.sqrt() * zs - sg * tau))], 1)
        dlab[at] = np.where(pts[at, 4:] > 0, np.nan, both)
    return [torch.from_numpy(lab), torch.from_numpy(dlab)]


def _layers(net, sizes, grad=False):
    out, o = [], 0
    for a, b in zip(sizes[:-1], sizes[1:]):
        t = torch.from_numpy(net).double().cuda()
        out.append((t[o:o + a * b].view(a, b).clone().requires_grad_(grad), t[o + a * b:o + a * b + b].clone().requires_grad_(grad)))
        o += a * b + b
    return out


def _exact_train(case, seed):
    net, sizes, x, y, g = _train_inputs(case, seed)
    par = _layers(net, sizes, True)
    h, y, g = (torch.from_numpy(a).double().cuda() for a in (x, y, g))
    dh = [torch.zeros_like(h).index_fill_(1, torch.tensor([DIRS[k]], device="cuda"), 1.0) for k in range(case["dirs"])]
    for i, (W, b) in enumerate(par):
        z, dz = h @ W + b, [t @ W for t in dh]
        if i == len(par) - 1:
            break
        s = torch.sigmoid(z)
        h, dh = z * s, [s * (1 + z * (1 - s)) * t for t in dz]
    parts = [((z[:, 0] - y) ** 2).mean()]
    for k in range(case["dirs"]):
        on = torch.isfinite(g[:, k])
        e = torch.where(on, SCALES[k] * dz[k][:, 0] - torch.nan_to_num(g[:, k]), torch.zeros_like(y))
        parts.append(WEIGHTS[k] * (e * e).mean())
    gr = torch.autograd.grad(sum(parts), [t for p in par for t in p])
    return [float(p.detach()) for p in parts], torch.cat([t.reshape(-1) for t in gr]).cpu()


def _exact_risk(case, seed):
    pf, ns, u = _portfolio(case, seed), case["scenarios"], case["under"]
    T = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    s0, sg = T(pf["s0"]), T(pf["sigma"])
    h, dt = pf["horizon"], 1.0 / 252
    scen = torch.arange(ns, dtype=torch.int64, device="cuda")
    z = _normals(0, (u + 3) // 4, (2 << 56) | scen, seed)[:u]
    L = T(np.linalg.cholesky(pf["corr"])) * (sg * math.sqrt(h))[:, None]
    S = s0[:, None] * torch.exp(((RATE - 0.5 * sg * sg) * h)[:, None] + L @ z)  # [under, scenarios]
    under, kind = torch.from_numpy(pf["under"]).long().cuda(), torch.from_numpy(pf["kind"]).cuda()
    K, H, pos = T(pf["strike"]), T(pf["barrier"]), T(pf["position"])
    days = np.rint(pf["maturity"] * 252).astype(int)
    knock = kind == 4
    if case["method"] == "surrogate":
        par = _layers(*_net(256, 4, seed + 1))

        def value(S, steps):  # S [options, n]
            f = torch.stack([S / K[:, None], sg[under][:, None].expand_as(S), (steps * dt)[:, None].expand_as(S),
                             torch.full_like(S, RATE), torch.where(knock, K / H, torch.zeros_like(K))[:, None].expand_as(S)], 2)
            x = (f - T(SHIFT)) / T(SLOPE)
            for i, (W, b) in enumerate(par):
                x = x @ W + b
                x = x * torch.sigmoid(x) if i < len(par) - 1 else x
            call = K[:, None] * x[:, :, 0]
            put = call - S + (K * torch.exp(-RATE * steps * dt))[:, None]
            out = torch.where((S >= H[:, None]), torch.zeros_like(S), call.clamp_min(0.0))
            return torch.where(knock[:, None], out, torch.where((kind == 1)[:, None], put, call))
        base = value(s0[under][:, None], T(days))[:, 0]
        size = max(1, (1 << 20) // len(K))
        pnl = torch.cat([pos @ (value(S[under][:, i:i + size], T(days - 1)) - base[:, None]) for i in range(0, ns, size)])
    else:
        def value(S1, streams, steps, paths):
            """Options x rows; streams [u, rows]: the first stream of each underlying's inner paths."""
            out = torch.empty((len(K), S1.shape[1]), dtype=torch.float64, device="cuda")
            a, b = (RATE - 0.5 * sg * sg) * dt, sg * math.sqrt(dt)
            size = max(1, (1 << 18) // paths)
            for k in range(u):
                mine = np.nonzero(pf["under"] == k)[0]
                top = int(steps[mine].max())
                for i in range(0, S1.shape[1], size):
                    s1 = S1[k, i:i + size]
                    n = (streams[k, i:i + size, None] + torch.arange(paths, device="cuda")).reshape(-1)
                    y = torch.zeros(n.numel(), dtype=torch.float64, device="cuda")
                    mx = torch.full_like(y, -math.inf)
                    at = {}
                    for j, z in enumerate(_steps(n, 1, top, seed)):
                        y = y + (a[k] + b[k] * z[0])
                        mx = torch.maximum(mx, y)
                        if (steps[mine] == j + 1).any():
                            at[j + 1] = (y, mx)
                    for o in mine:
                        y1, m1 = (s1[:, None] * torch.exp(t.view(len(s1), paths)) for t in at[int(steps[o])])
                        f = (K[o] - y1 if pf["kind"][o] == 1 else y1 - K[o]).clamp_min(0.0)
                        if pf["kind"][o] == 4:
                            f = torch.where((m1 >= H[o]) | (s1 >= H[o])[:, None], torch.zeros_like(f), f)
                        out[o, i:i + size] = math.exp(-RATE * dt * steps[o]) * f.mean(1)
            return out
        ks = torch.arange(u, dtype=torch.int64, device="cuda")[:, None]
        base = value(s0[:, None], (5 << 56) | (ks << 24), days, 1 << 16)[:, 0]
        pnl = pos @ (value(S, (3 << 56) | ((scen[None, :] * u + ks) << 16), days - 1, case["inner"]) - base[:, None])
    loss = (-pnl).sort(descending=True)[0]
    var = loss[max(1, math.ceil(0.01 * ns - 1e-9)) - 1]
    tail = loss[loss > var]
    return dict(var=float(var), cvar=float(tail.mean()) if len(tail) else float(var), base_value=float(pos @ base),
                n_tail=None)


def exact(case, seed):
    what = case["what"]
    if what == "risk" and case["method"] == "surrogate" and case["scenarios"] * case["under"] * case["per_under"] > 1 << 25:
        return None  # the network in 64 bits on more rows takes too long
    with torch.no_grad() if what not in ("grad", "train") else torch.enable_grad():
        return dict(price=_exact_price, heston=_exact_heston, grad=_exact_grad, labels=_exact_labels,
                    train=_exact_train, risk=_exact_risk)[what](case, seed)
