"""The calls this library is timed on: their inputs, one pass of each through the
public Python entry points, the work a pass cannot do without, and its values in FP64.

A case is a dict of plain values:
  call    price | fd | adjoint | book | lsm | basket (the entry point)
  model   base (the single-option model, moved a little per seed, as a re-pricing on new
          market data moves it) | drawn (parameters over the book's ranges, the Feller
          condition often broken)
  strikes number of strikes, evenly spaced on K/S0 in [0.7, 1.3]; one strike is at the money
  steps, paths, put, scheme (qe | qem)
  greeks  fd: comma-separated Greeks; book: "adjoint" or ""
  options, spread  book: number of options; spread true: each option its own steps and paths,
          log-uniform in [16, steps] and [paths / 64, paths]; false: all steps x paths
  every   lsm: steps between exercise dates
  assets  basket: correlated assets
The FP64 values follow the scheme's published definition (Andersen's QE on Philox4x32-10
draws), written here in plain torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2402_12111_gb300 as simr

BASE = dict(S0=100.0, r=0.05, T=1.0, v0=0.04, kappa=1.5, theta=0.04, sigma=0.3, rho=-0.7)
BENCH_GREEKS = "delta,gamma,vega,theta,rho"
MODEL_GREEKS = "delta,vega,rho,kappa,lrvar,volvol,corr"
DEFAULTS = dict(call="price", model="base", strikes=1, steps=64, paths=65536, put=False, scheme="qe", greeks="",
                options=1, spread=False, every=1, assets=1)


def _case(name, **kw):
    return {"name": name, **DEFAULTS, **kw}


def listed():
    return [
        # three strikes of a short-dated option: what a quoting loop asks for; launch latency
        _case("price_quote", strikes=3, steps=16, paths=8192),
        # one option with its hedge Greeks, the library's default size
        _case("fd_single", call="fd", steps=64, paths=65536, greeks="delta,gamma,vega"),
        # a strike grid of one underlying at daily steps: the calibration / re-pricing call
        _case("price_grid", strikes=32, steps=252, paths=1 << 20),
        # the benchmark step: the same grid with five bump-and-revalue Greeks
        _case("fd_grid", call="fd", strikes=32, steps=252, paths=1 << 20, greeks=BENCH_GREEKS),
        # every model sensitivity by bumping (11 scenarios), ragged strike, step and path counts
        _case("fd_model_ragged", call="fd", strikes=21, steps=365, paths=250001, put=True, greeks=MODEL_GREEKS),
        # the grid's seven sensitivities by the pathwise adjoint
        _case("adjoint_grid", call="adjoint", strikes=32, steps=252, paths=1 << 20),
        # martingale-corrected puts on two strike tiles, odd steps, ragged paths
        _case("price_qem_ragged", model="drawn", strikes=40, steps=101, paths=300007, put=True, scheme="qem"),
        # the paper's smallest problem, 5 assets x 126 steps x 25,000 paths, as a book
        _case("book_tiny", call="book", model="drawn", options=5, steps=126, paths=25000),
        # a desk's heterogeneous book with adjoint Greeks
        _case("book_adjoint", call="book", model="drawn", options=64, spread=True, steps=512, paths=1 << 20,
              greeks="adjoint"),
        # Bermudan put exercisable daily: the Longstaff-Schwartz benchmark
        _case("lsm_daily", call="lsm", steps=252, paths=1 << 20, put=True),
        # eight correlated assets on the strike grid
        _case("basket8", call="basket", model="drawn", assets=8, strikes=32, steps=252, paths=1 << 18),
        # one underlying of the largest configured run: 1,024 steps x 2^26 paths, adjoint
        _case("adjoint_headline", call="adjoint", model="drawn", strikes=32, steps=1024, paths=1 << 26),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    c = dict(DEFAULTS)
    c["call"] = rng.choice(["price", "price", "fd", "fd", "adjoint", "adjoint", "book", "lsm", "basket"])
    c["model"] = rng.choice(["base", "drawn"])
    c["put"] = rng.random() < 0.5
    c["strikes"] = rng.choice([1, rng.randint(2, 31), 32, rng.randint(33, 64)])
    c["steps"] = _log_int(rng, 8, 1024)
    c["paths"] = _log_int(rng, 4096, 1 << 22)
    c["scheme"] = rng.choice(["qe", "qe", "qem"])
    if c["call"] == "fd":
        c["greeks"] = rng.choice(["delta,gamma,vega", "vega", BENCH_GREEKS, MODEL_GREEKS])
    elif c["call"] == "book":
        c.update(strikes=1, model="drawn", options=_log_int(rng, 2, 128), spread=rng.random() < 0.7,
                 greeks=rng.choice(["", "adjoint"]), steps=_log_int(rng, 16, 512))
        c["paths"] = _log_int(rng, 16384, 1 << (20 if c["spread"] else 18))
    elif c["call"] == "lsm":
        c["every"] = rng.choice([1, 1, 5, 21])
        c.update(strikes=1, model="base", steps=c["every"] * max(2, _log_int(rng, 8, 252) // c["every"]),
                 paths=_log_int(rng, 16384, 1 << 20))
    elif c["call"] == "basket":
        c.update(model="drawn", assets=rng.randint(2, 12), steps=_log_int(rng, 8, 252), paths=_log_int(rng, 4096, 1 << 19))
    return c


# ---------------------------------------------------------------- inputs ----
def _model(case, rng):
    if case["model"] == "drawn":
        return dict(S0=100.0, r=rng.uniform(0.0, 0.06), T=rng.uniform(0.1, 3.0), v0=rng.uniform(0.01, 0.09),
                    kappa=rng.uniform(0.5, 5.0), theta=rng.uniform(0.01, 0.09), sigma=rng.uniform(0.1, 1.0),
                    rho=rng.uniform(-0.95, 0.0))
    m = {k: v * rng.uniform(0.97, 1.03) for k, v in BASE.items()}
    m["T"] = BASE["T"]
    return m


def _inputs(case, seed):
    """Everything the seed decides, on the host: models, strikes, weights, the Philox seed."""
    rng = random.Random(seed)
    s = dict(seed=rng.randrange(1, 1 << 48))
    n = case["options"] if case["call"] == "book" else case["assets"]
    s["models"] = [_model(case, rng) for _ in range(n)]
    m = s["models"][0]
    nk = case["strikes"]
    s["strikes"] = [m["S0"] * (0.7 + 0.6 * i / (nk - 1)) if nk > 1 else m["S0"] for i in range(nk)]
    if case["call"] == "book":
        s["book"] = []
        for mk in s["models"]:
            steps, paths = case["steps"], case["paths"]
            if case["spread"]:
                steps = _log_int(rng, min(16, steps), steps)
                paths = _log_int(rng, max(1, paths // 64), paths)
            s["book"].append(dict(model=mk, K=100.0 * rng.uniform(0.7, 1.3), is_put=rng.random() < 0.5, steps=steps,
                                  paths=paths))
    if case["call"] == "basket":
        for mk in s["models"]:
            mk["T"], mk["r"] = 1.0, 0.03
        g = np.array([[rng.gauss(0.0, 1.0) for _ in range(n + 2)] for _ in range(n)])
        cov = g @ g.T
        c = cov / np.sqrt(np.outer(np.diag(cov), np.diag(cov)))
        c = 0.5 * (c + c.T)
        np.fill_diagonal(c, 1.0)
        s["corr"], s["weights"] = c, np.full(n, 1.0 / n)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    s["K"] = torch.tensor(s["strikes"], dtype=torch.float64, device="cuda")
    s["names"] = tuple(g for g in case["greeks"].split(",") if g)
    simr.load()
    return s


def run(s):
    if s["case"]["scheme"] == "qem":
        with simr.scheme("qem"):
            return _run(s)
    return _run(s)


def _run(s):
    c, m = s["case"], s["models"][0]
    if c["call"] == "price":
        return simr.price(m, s["K"], c["put"], c["steps"], c["paths"], s["seed"])
    if c["call"] == "fd":
        return simr.greeks_fd(m, s["K"], c["put"], c["steps"], c["paths"], s["seed"], greeks=s["names"])
    if c["call"] == "adjoint":
        return simr.greeks_adjoint(m, s["K"], c["put"], c["steps"], c["paths"], s["seed"])
    if c["call"] == "book":
        return simr.batch(s["book"], seed=s["seed"], adjoint=c["greeks"] == "adjoint")
    if c["call"] == "lsm":
        return simr.lsm_price(m, s["strikes"][0], c["put"], c["steps"], c["every"], c["paths"], s["seed"])[:2]
    return simr.basket_price(s["models"], s["corr"], s["weights"], s["K"], c["put"], c["steps"], c["paths"], s["seed"])


# ------------------------------------------------------------------ work ----
RESIM = {"vega": "v0", "theta": "T", "kappa": "kappa", "lrvar": "theta", "volvol": "sigma", "corr": "rho"}


def _path_steps(case, seed=0):
    """Path-steps of a pass (a spread book's: their mean over the ranges)."""
    if case["call"] == "book" and case["spread"]:
        a, b = min(16, case["steps"]), case["steps"]
        p, q = max(1, case["paths"] // 64), case["paths"]
        mean = lambda lo, hi: (hi - lo) / math.log(hi / lo) if hi > lo else lo  # noqa: E731
        return case["options"] * mean(a, b) * mean(p, q)
    return case["steps"] * case["paths"] * (case["options"] if case["call"] == "book" else case["assets"])


def work(case):
    """Flops of the method (a fused multiply-add is 2): 44 per path-step for the two inverse
    normals, 23 per simulated scenario for the QE and log-spot steps, 51 for the adjoint's
    reverse step; a basket's correlation 2 per lower-triangle entry.  Bytes: strikes in,
    results out; Longstaff-Schwartz also writes and reads S and v at every date."""
    ps, nk = _path_steps(case), case["strikes"]
    names = [g for g in case["greeks"].split(",") if g]
    per, out = 44 + 23, 2 * nk
    if case["call"] == "fd":
        per, out = 44 + 23 * (1 + 2 * sum(g in RESIM for g in names)), nk * (1 + len(names))
    adjoint = case["call"] == "adjoint" or case["greeks"] == "adjoint"
    if adjoint:
        per, out = per + 51, out + 7 * nk
    if case["call"] == "book":
        out *= case["options"]
    if case["call"] == "basket":
        per += case["assets"] + 1
    nbytes = 8.0 * (nk + out)
    if case["call"] == "lsm":
        nbytes += 16.0 * (case["steps"] // case["every"]) * case["paths"]
    return {"bytes": nbytes, "flops": float(per) * ps}


# ----------------------------------------------------- the values in FP64 ----
MASK = 0xFFFFFFFF


def _mulhilo(a: int, x):
    """High and low words of a * x for 32-bit words held in int64."""
    p0, p1 = (x & 0xFFFF) * a, (x >> 16) * a
    mid = (p0 >> 16) + (p1 & 0xFFFF)
    return (p1 >> 16) + (mid >> 16), ((mid & 0xFFFF) << 16) | (p0 & 0xFFFF)


def _philox(seed, pair, path, option):
    """The four words of Philox4x32-10 for counter (pair, path lo, path hi, option), int64."""
    k0, k1 = seed & MASK, (seed >> 32) & MASK
    c = [torch.full_like(path, pair), path & MASK, path >> 32, torch.full_like(path, option)]
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, c[0])
        h1, l1 = _mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return c


def _draws(seed, n, path, option):
    """(U_V, Phi^-1(U_V), Phi^-1(U_X)) of step n for the paths; u = ((word >> 9) + 1/2) 2^-23."""
    w = _philox(seed, n // 2, path, option)[2 * (n % 2):2 * (n % 2) + 2]
    uv, ux = (((x >> 9).double() + 0.5) * 2.0 ** -23 for x in w)
    return uv, torch.special.ndtri(uv), torch.special.ndtri(ux)


def _step(m, steps, qem, v, uv, zv, zx):
    """One step of Andersen's QE (psi_c = 1.5, gamma1 = gamma2 = 1/2), QE-M with qem: (v', x' - x).
    m holds numbers or per-path tensors; differentiable with the branch held fixed."""
    exp, sqrt = (lambda a: a.exp() if torch.is_tensor(a) else math.exp(a)), \
                (lambda a: a.sqrt() if torch.is_tensor(a) else math.sqrt(a))
    dt = m["T"] / steps
    kap, th, sg, rho = m["kappa"], m["theta"], m["sigma"], m["rho"]
    E = exp(-kap * dt)
    mean = th + (v - th) * E
    s2 = v * sg * sg * E * (1 - E) / kap + th * sg * sg * (1 - E) * (1 - E) / (2 * kap)
    psi = s2 / (mean * mean)
    quad = psi <= 1.5
    t = torch.where(quad, 2.0 / torch.where(quad, psi, 1.0), 2.0)
    b2 = t - 1.0 + torch.sqrt(t * (t - 1.0))
    a = mean / (1.0 + b2)
    pe = torch.where(quad, 0.5, (psi - 1.0) / (psi + 1.0))  # the atom's mass
    beta = (1.0 - pe) / mean
    up = ~quad & (uv > pe)
    ve = torch.where(up, torch.log(torch.where(up, (1.0 - pe) / (1.0 - uv), 1.0)) / beta, 0.0)
    vn = torch.where(quad, a * (torch.sqrt(b2) + zv) ** 2, ve)
    K1 = 0.5 * dt * (kap * rho / sg - 0.5) - rho / sg
    K2 = 0.5 * dt * (kap * rho / sg - 0.5) + rho / sg
    K3 = 0.5 * dt * (1.0 - rho * rho)
    K0 = -rho * kap * th * dt / sg
    if qem:
        A = K2 + 0.5 * K3
        okq = quad & (2.0 * A * a < 1.0)
        oke = ~quad & (A < beta)
        aq = torch.where(okq, 2.0 * A * a, 0.0)
        lnq = 0.5 * aq * b2 / (1.0 - aq) - 0.5 * torch.log1p(-aq)
        we = torch.where(oke, A / beta, 0.0)
        lne = torch.log(pe + (1.0 - pe) / (1.0 - we))
        ok = okq | oke
        K0 = torch.where(ok, -torch.where(quad, lnq, lne) - (K1 + 0.5 * K3) * v, K0)
    s = v + vn
    pos = s > 0
    root = sqrt(K3) * torch.where(pos, torch.sqrt(torch.where(pos, s, 1.0)), 0.0)
    return vn, m["r"] * dt + K0 + K1 * v + K2 * vn + root * zx


def _terminal(models, steps, seed, path, option=0, qem=False, record=0):
    """x_T of each model on common draws; with record: the lists of (x, v) of the first model at
    every record-th step."""
    v = [torch.zeros_like(path, dtype=torch.float64) + m["v0"] for m in models]
    x = [torch.zeros_like(path, dtype=torch.float64) for _ in models]
    kept = []
    for n in range(steps):
        uv, zv, zx = _draws(seed, n, path, option)
        for j, m in enumerate(models):
            v[j], dx = _step(m, steps, qem, v[j], uv, zv, zx)
            x[j] = x[j] + dx
        if record and (n + 1) % record == 0:
            kept.append((x[0], v[0]))
    return kept if record else x


def _payoff(put, S, K):
    return torch.clamp(K - S if put else S - K, min=0.0)


def _estimate(s1, s2, disc, n):
    mean = s1 / n
    var = (s2 / n - mean * mean) / (n - 1) if n > 1 else torch.zeros_like(mean)
    return disc * mean, disc * torch.sqrt(torch.clamp(var, min=0.0))


def _chunks(paths, size):
    for a in range(0, paths, size):
        yield torch.arange(a, min(a + size, paths), dtype=torch.int64, device="cuda")


def _price64(m, strikes, put, steps, paths, seed, option, qem):
    s = torch.zeros(2, len(strikes), dtype=torch.float64, device="cuda")
    for path in _chunks(paths, 1 << 20):
        S = m["S0"] * torch.exp(_terminal([m], steps, seed, path, option, qem)[0])
        for k, K in enumerate(strikes):
            f = _payoff(put, S, K)
            s[0, k] += f.sum()
            s[1, k] += (f * f).sum()
    return _estimate(s[0], s[1], math.exp(-m["r"] * m["T"]), paths)


def _fd64(m, strikes, put, steps, paths, seed, names, qem, rel=1e-4):
    """Prices and central differences on common draws, columns in the library's order."""
    order = [g for g in ("delta", "gamma", "vega", "theta", "rho", "kappa", "lrvar", "volvol", "corr") if g in names]
    models = [m]
    for g in order:
        if g in RESIM:
            h = rel if g == "corr" else rel * m[RESIM[g]]
            models += [dict(m, **{RESIM[g]: m[RESIM[g]] + h}), dict(m, **{RESIM[g]: m[RESIM[g]] - h})]
    disc = lambda q: math.exp(-q["r"] * q["T"])  # noqa: E731
    p = torch.zeros(len(strikes), dtype=torch.float64, device="cuda")
    g = torch.zeros(len(strikes), len(order), dtype=torch.float64, device="cuda")
    for path in _chunks(paths, 1 << 18):
        x = _terminal(models, steps, seed, path, 0, qem)
        S = [m["S0"] * torch.exp(xi) for xi in x]
        for k, K in enumerate(strikes):
            f = lambda Sx: _payoff(put, Sx, K).sum()  # noqa: E731
            p[k] += disc(m) * f(S[0]) / paths
            j = 1
            for i, name in enumerate(order):
                if name in RESIM:
                    h = rel if name == "corr" else rel * m[RESIM[name]]
                    d = (disc(models[j]) * f(S[j]) - disc(models[j + 1]) * f(S[j + 1])) / (2 * h)
                    d, j = (-d if name == "theta" else d), j + 2
                elif name == "delta":
                    d = disc(m) * (f(S[0] * (1 + rel)) - f(S[0] * (1 - rel))) / (2 * rel * m["S0"])
                elif name == "gamma":
                    d = disc(m) * (f(S[0] * (1 + rel)) - 2 * f(S[0]) + f(S[0] * (1 - rel))) / (rel * m["S0"]) ** 2
                else:
                    h = rel * m["r"]
                    up, dn = math.exp(h * m["T"]), math.exp(-h * m["T"])
                    d = disc(m) * (dn * f(S[0] * up) - up * f(S[0] * dn)) / (2 * h)
                g[k, i] += d / paths
    return p, g


def _adjoint64(m, strikes, put, steps, paths, seed, option, qem):
    """Price, standard error and the seven pathwise derivatives (S0, v0, kappa, theta, sigma, rho, r)."""
    s = torch.zeros(9, len(strikes), dtype=torch.float64, device="cuda")
    for path in _chunks(paths, max(1024, min(1 << 18, (1 << 25) // steps))):
        q = {k: torch.full(path.shape, m[k], dtype=torch.float64, device="cuda", requires_grad=True)
             for k in ("v0", "kappa", "theta", "sigma", "rho")}
        x = _terminal([dict(m, **q)], steps, seed, path, option, qem)[0]
        dx = torch.autograd.grad(x.sum(), list(q.values()))
        S = m["S0"] * torch.exp(x.detach())
        for k, K in enumerate(strikes):
            f = _payoff(put, S, K)
            w = torch.where(S < K, -S, 0.0) if put else torch.where(S > K, S, 0.0)  # f'(S) S
            cols = [f, f * f, w / m["S0"]] + [w * d for d in dx] + [m["T"] * (w - f)]
            s[:, k] += torch.stack([c.sum() for c in cols])
    disc = math.exp(-m["r"] * m["T"])
    price, err = _estimate(s[0], s[1], disc, paths)
    return price, err, (disc * s[2:] / paths).T.contiguous()


def _lsm64(m, K, put, steps, every, paths, seed, qem):
    """Longstaff-Schwartz on quadratics of (S, v), in-the-money paths, 12 of them at least."""
    path = torch.arange(paths, dtype=torch.int64, device="cuda")
    kept = _terminal([m], steps, seed, path, 0, qem, record=every)
    dates, dt = len(kept), m["T"] / len(kept)
    cash = _payoff(put, m["S0"] * torch.exp(kept[-1][0]), K)
    for j in range(dates - 2, -1, -1):
        cash = cash * math.exp(-m["r"] * dt)
        x, v = kept[j]
        S = m["S0"] * torch.exp(x)
        h = _payoff(put, S, K)
        itm = h > 0
        if int(itm.sum()) < 12:
            continue
        a, b = (S[itm] - S.mean()) / S.std(), (v[itm] - v.mean()) / v.std()
        phi = torch.stack([torch.ones_like(a), a, a * a, b, a * b, b * b], 1)
        fit = phi @ torch.linalg.solve(phi.T @ phi, phi.T @ cash[itm])
        cash[itm] = torch.where(h[itm] > fit, h[itm], cash[itm])
    cash = cash * math.exp(-m["r"] * dt)
    return _estimate(cash.sum().view(1), (cash * cash).sum().view(1), 1.0, paths)


def _basket64(s, put, steps, paths, qem):
    models = s["models"]
    low = np.linalg.cholesky(s["corr"])
    t = torch.zeros(2, len(s["strikes"]), dtype=torch.float64, device="cuda")
    for path in _chunks(paths, 1 << 20):
        v = [torch.full(path.shape, m["v0"], dtype=torch.float64, device="cuda") for m in models]
        x = [torch.zeros_like(v[0]) for _ in models]
        for n in range(steps):
            d = [_draws(s["seed"], n, path, k) for k in range(len(models))]
            for k, m in enumerate(models):
                z = sum(low[k, j] * d[j][2] for j in range(k + 1))
                v[k], dx = _step(m, steps, qem, v[k], d[k][0], d[k][1], z)
                x[k] = x[k] + dx
        B = sum(w * m["S0"] * torch.exp(xk) for w, m, xk in zip(s["weights"], models, x))
        for k, K in enumerate(s["strikes"]):
            f = _payoff(put, B, K)
            t[0, k] += f.sum()
            t[1, k] += (f * f).sum()
    return _estimate(t[0], t[1], math.exp(-models[0]["r"] * models[0]["T"]), paths)


# Seconds of the FP64 evaluation: a path-step's arithmetic and a step's launches.
PATH_STEP_S, STEP_S = 1.5e-9, 1.5e-3


def _exact_seconds(case, s):
    scen = 1 + 2 * sum(g in RESIM for g in case["greeks"].split(","))
    weight = 5.0 if case["call"] == "adjoint" or case["greeks"] == "adjoint" else 0.4 + 0.6 * scen
    jobs = [(o["steps"], o["paths"]) for o in s["book"]] if case["call"] == "book" else \
        [(case["steps"], case["paths"])] * case["assets"]
    size = {"fd": 1 << 18}.get(case["call"], 1 << 20)
    total = 0.0
    for steps, paths in jobs:
        n = max(1024, min(1 << 18, (1 << 25) // steps)) if weight == 5.0 else size
        total += weight * steps * (paths * PATH_STEP_S + -(-paths // n) * STEP_S)
    dates = case["steps"] // case["every"] if case["call"] == "lsm" else 0  # their regressions
    return total * (2.0 if case["call"] == "basket" else 1.0) + dates * case["paths"] * 3.5e-8


def exact(case, seed):
    s = _inputs(case, seed)
    if _exact_seconds(case, s) > 20.0:
        return None
    qem, put, steps, paths = case["scheme"] == "qem", case["put"], case["steps"], case["paths"]
    m, K, sd = s["models"][0], s["strikes"], s["seed"]
    if case["call"] == "price":
        return _price64(m, K, put, steps, paths, sd, 0, qem)
    if case["call"] == "fd":
        return _fd64(m, K, put, steps, paths, sd, case["greeks"].split(","), qem)
    if case["call"] == "adjoint":
        return _adjoint64(m, K, put, steps, paths, sd, 0, qem)
    if case["call"] == "lsm":
        return _lsm64(m, K[0], put, steps, case["every"], paths, sd, qem)
    if case["call"] == "basket":
        return _basket64(s, put, steps, paths, qem)
    fn = _adjoint64 if case["greeks"] == "adjoint" else _price64
    rows = [fn(o["model"], [o["K"]], o["is_put"], o["steps"], o["paths"], sd, i, qem) for i, o in enumerate(s["book"])]
    cols = [torch.cat([r[k] for r in rows]) for k in range(len(rows[0]))]
    return (*cols, None) if len(cols) == 2 else tuple(cols)
