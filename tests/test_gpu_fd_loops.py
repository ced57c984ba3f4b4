"""The step loops of the bump-and-revalue kernels at the counts where a prologue, an odd
last step or a lone step can go wrong: 1, 2, 3 and 5 steps, and 4,092 / 4,095 (the last
with a table of the step pairs' counters, and without one); with step 0 split off, and
with a bump that carries it across the QE threshold, where it is not.

Loops over the same steps form the same FP32 sums of 32 paths; only the order of their
FP64 additions may differ: 1e-11 of a column's largest value.
"""
import math

import numpy as np
import pytest
import torch

import oracle
import test_gpu_parity as parity
import workloads

pytestmark = pytest.mark.gpu

CFG = dict(workloads.BASE_MODEL)
K3 = np.array([90.0, 100.0, 110.0])
GREEKS = {3: ("vega",), 5: ("vega", "theta"), 7: ("vega", "theta", "kappa"), 9: ("vega", "theta", "kappa", "lrvar"),
          11: ("vega", "kappa", "lrvar", "volvol", "corr"), 13: ("vega", "theta", "kappa", "lrvar", "volvol", "corr")}


@pytest.fixture(scope="module")
def simr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2402_12111_gb300 as simr

    simr.load()
    return simr


def _psi(m, steps):
    dt = m["T"] / steps
    E = math.exp(-m["kappa"] * dt)
    mean = m["theta"] + (m["v0"] - m["theta"]) * E
    s2 = m["sigma"] ** 2 * (m["v0"] * E * (1 - E) / m["kappa"] + m["theta"] * (1 - E) ** 2 / (2 * m["kappa"]))
    return s2 / mean ** 2


def _model(steps, split):
    """With split: step 0 on one side of psi = 1.5 for every bump of 1e-2; without: a bump of
    v0 or T carries it across (the base's psi 0.1% above; FP32 resolves 1e-6)."""
    if split:
        return dict(CFG)
    m = dict(CFG, v0=0.16, kappa=0.5, sigma=1.0)
    m["sigma"] = math.sqrt(1.5015 / _psi(m, steps))
    sides = {_psi(dict(m, v0=m["v0"] * (1 + h)), steps) > 1.5 for h in (-1e-2, 1e-2)}
    assert sides == {True, False} and _psi(m, steps) > 1.5 * 1.0005
    return m


def _dev(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float64), device="cuda")


def _same(a, b):
    for x, y in zip(a, b):
        scale = y.abs().amax(dim=0, keepdim=True).clamp_min(1e-300)
        assert torch.all((x - y).abs() <= 1e-11 * scale), float(((x - y).abs() / scale).max())


@pytest.mark.parametrize("scheme", ["qe", "qem"])
@pytest.mark.parametrize("split", [True, False])
@pytest.mark.parametrize("scen", list(GREEKS))
@pytest.mark.parametrize("steps", [1, 2, 3, 5, 4095])
def test_a_strike_alone_equals_the_strike_in_a_grid(simr, steps, scen, split, scheme):
    # one strike: two steps an iteration (3 and 5 scenarios pipelined); a tile of strikes:
    # one step an iteration from 7 scenarios on and under QE-M
    if steps == 4095 and not split:
        pytest.skip("a step that short crosses the threshold at sigma > 10 only")
    m, paths = _model(steps, split), 5000 if steps < 100 else 700
    with simr.scheme(scheme):
        grid = simr.greeks_fd(m, _dev(K3), False, steps, paths, 7, greeks=GREEKS[scen], rel_bump=1e-2)
        alone = [simr.greeks_fd(m, _dev([k]), False, steps, paths, 7, greeks=GREEKS[scen], rel_bump=1e-2) for k in K3]
    _same(grid, [torch.cat([a[i] for a in alone]) for i in range(2)])


@pytest.mark.parametrize("steps", [760, 761, 762])
def test_eleven_scenarios_at_the_step_count_that_changes_the_loop(simr, steps):
    # a tile of strikes under QE: one step an iteration up to 760 steps, two beyond
    grid = simr.greeks_fd(CFG, _dev(K3), False, steps, 700, 7, greeks=GREEKS[11], rel_bump=1e-2)
    alone = [simr.greeks_fd(CFG, _dev([k]), False, steps, 700, 7, greeks=GREEKS[11], rel_bump=1e-2) for k in K3]
    _same(grid, [torch.cat([a[i] for a in alone]) for i in range(2)])


@pytest.mark.parametrize("split", [True, False])
@pytest.mark.parametrize("n_strikes", [1, 3])
@pytest.mark.parametrize("scen", [3, 5])
@pytest.mark.parametrize("steps", [1, 2, 3, 4, 5, 4092, 4095])
def test_pipelined_scenarios_equal_the_plain_loop(simr, steps, scen, n_strikes, split):
    # the 3- and 5-scenario loop draws a step ahead; the same Greeks asked beside one more
    # run through the 13-scenario kernel's loop, which does not
    if steps > 1000 and not split:
        pytest.skip("a step that short crosses the threshold at sigma > 10 only")
    m, paths, K = _model(steps, split), 5000 if steps < 100 else 700, _dev(K3[:n_strikes])
    a = simr.greeks_fd(m, K, True, steps, paths, 9, greeks=GREEKS[scen], rel_bump=1e-2)
    b = simr.greeks_fd(m, K, True, steps, paths, 9, greeks=GREEKS[9], rel_bump=1e-2)
    _same(a, (b[0], b[1][:, :len(GREEKS[scen])]))


@pytest.mark.parametrize("split", [True, False])
@pytest.mark.parametrize("n_strikes", [1, 3])
@pytest.mark.parametrize("scen", [3, 5])
@pytest.mark.parametrize("steps", [1, 2, 3, 5])
def test_pipelined_scenarios_match_the_oracle(simr, steps, scen, n_strikes, split):
    # the bounds of the Greeks' parity test; and for a path whose QE decision lies within
    # 5e-6 of its threshold in any of a Greek's scenarios (FP32 may take the other branch:
    # t carries a few roundings of 6e-8) a payoff as large as any seen
    m, paths, h, K = _model(steps, split), 1 << 14, 1e-2, K3[:n_strikes]
    p, g = simr.greeks_fd(m, _dev(K), False, steps, paths, 11, greeks=GREEKS[scen], rel_bump=h)
    p, g = p.cpu().numpy(), g.cpu().numpy()
    po, go = oracle.greeks_fd(m, K, False, steps, paths, 11, h, sum(parity.ORACLE_BITS[x] for x in GREEKS[scen]))

    def close(field):
        n, top = 0, 0.0
        for f in (1 - h, 1.0, 1 + h):
            x, _, mg = oracle.terminal(dict(m, **{field: m[field] * f}), steps, 11, 0, paths)
            n, top = n + int((mg < 5e-6).sum()), max(top, m["S0"] * math.exp(x.max()))
        return n * np.maximum(top - K, 0.0) / paths

    assert np.all(np.abs(p - po) <= 1e-5 * np.abs(po) + close("v0") + 1e-12)
    for j, name in enumerate(GREEKS[scen]):
        tol = parity._greek_tol(name, go[:, j], h, steps, paths, m) + \
            close({"vega": "v0", "theta": "T"}[name]) / parity.BUMPS[name](m, h)
        assert np.all(np.abs(g[:, j] - go[:, j]) <= tol), (name, g[:, j] - go[:, j], tol)
