"""The path kernels' items: a block's batches handed to its warps one item at a time,
the item's rows and the two-level sum over blocks, and the step pairs' counter table.

A launch over a path range equals the sum of launches over its parts: the parts
start on multiples of 64 paths, so they form the same FP32 sums of 32 (pricing:
64) paths, and only the order of the FP64 additions differs.  The bound is
n_sums * 2^-53 relative to the sum of the magnitudes for at most 2^16 FP32 sums,
7e-12, taken as 1e-11 of the column's largest value.
"""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def simr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2402_12111_gb300 as simr

    simr.load()
    return simr


def _sums(simr, K, steps, begin, count, greeks=()):
    s = simr.path_sums(dict(workloads.BASE_MODEL), K, False, steps, begin, count, seed=11, greeks=greeks)
    return s.cpu().numpy()


def _check(whole, parts):
    got = np.sum(parts, axis=0)
    scale = np.maximum(np.abs(whole).max(axis=0, keepdims=True), 1e-300)
    assert np.all(np.abs(whole - got) <= 1e-11 * scale), np.max(np.abs(whole - got) / scale)


SMS = 152
# one path; one batch short of, at and past a batch, a block's warps and the grid;
# several items a warp; FP64 levels before the single batches
PATHS = [1, 63, 64, 65, 64 * SMS - 1, 64 * SMS + 1, 64 * SMS * 28 + 33, 64 * SMS * 90 + 5]


@pytest.mark.parametrize("paths", PATHS)
@pytest.mark.parametrize("n_strikes", [1, 32, 33])
def test_prices_over_a_range_are_the_sum_of_its_parts(simr, paths, n_strikes):
    K = torch.linspace(70.0, 130.0, n_strikes, dtype=torch.float64, device="cuda") if n_strikes > 1 else \
        torch.tensor([100.0], dtype=torch.float64, device="cuda")
    cut = paths // 3 // 64 * 64
    parts = [_sums(simr, K, 3, 0, cut)] if cut else []
    _check(_sums(simr, K, 3, 0, paths), parts + [_sums(simr, K, 3, cut, paths - cut)])


@pytest.mark.parametrize("greeks,n_strikes,paths", [
    (("delta", "gamma", "vega"), 1, 32 * SMS * 40 + 7),
    (("delta", "gamma", "vega", "theta", "rho"), 32, 32 * SMS * 300 + 9),  # levels of FP64 rows, then FP32 ones
    (("delta", "vega", "kappa"), 256, 32 * SMS * 40 + 1),                  # few rows fit: wider items to the end
    (tuple("delta gamma vega theta rho kappa lrvar volvol corr".split()), 40, 32 * SMS * 9 + 31),
])
def test_greeks_over_a_range_are_the_sum_of_its_parts(simr, greeks, n_strikes, paths):
    K = torch.linspace(80.0, 120.0, n_strikes, dtype=torch.float64, device="cuda")
    cut = paths // 2 // 64 * 64
    _check(_sums(simr, K, 2, 0, paths, greeks),
           [_sums(simr, K, 2, 0, cut, greeks), _sums(simr, K, 2, cut, paths - cut, greeks)])


def test_many_strikes_leave_room_for_few_rows(simr):
    # 1,024 strikes: 16 KB a row; the price call against the sum of 256-strike calls
    K = torch.linspace(60.0, 140.0, 1024, dtype=torch.float64, device="cuda")
    paths = 64 * SMS * 30 + 11
    p, se = simr.price(dict(workloads.BASE_MODEL), K, False, 2, paths, 11)
    for a in range(0, 1024, 256):
        q, sq = simr.price(dict(workloads.BASE_MODEL), K[a:a + 256], False, 2, paths, 11)
        torch.testing.assert_close(p[a:a + 256], q, rtol=1e-11, atol=1e-11)
        torch.testing.assert_close(se[a:a + 256], sq, rtol=1e-9, atol=1e-11)


@pytest.mark.parametrize("greeks", [(), ("delta", "vega")])
def test_paths_across_a_multiple_of_2_to_the_32(simr, greeks):
    # the paths' high counter words differ: no table; either side alone has one
    K = torch.tensor([95.0, 105.0], dtype=torch.float64, device="cuda")
    b = (1 << 32) - 192
    _check(_sums(simr, K, 5, b, 500, greeks), [_sums(simr, K, 5, b, 192, greeks), _sums(simr, K, 5, 1 << 32, 308, greeks)])


@pytest.mark.parametrize("scheme", ["qe", "qem"])
@pytest.mark.parametrize("model", [dict(), dict(sigma=1.0, rho=-0.9, kappa=0.5, T=2.0)])  # Feller ratio 1.3, 0.04
@pytest.mark.parametrize("steps", [1, 2, 3, 8, 4092, 4095])  # the shortest pipelines; the table's last entry and none
def test_step_counts_match_the_per_path_simulation(simr, steps, scheme, model):
    # the pipelined two-path loop against the terminal states of the one-path loop:
    # the same path, so S_T agrees to the rounding of x_T to one float, 2^-24
    # max(1, |x|), and the payoffs' mean to 1e-6 of the mean spot (200 paths of
    # either sign); any wrong draw or branch moves a path by 1e-3 and more
    m = dict(workloads.BASE_MODEL, **model)
    K = torch.tensor([95.0, 105.0], dtype=torch.float64, device="cuda")
    with simr.scheme(scheme):
        p, _ = simr.price(m, K, False, steps, 200, 5)
        x, _ = simr.paths_terminal(m, steps, 0, 200, seed=5)
    S = m["S0"] * torch.exp(x.double())
    ref = np.exp(-m["r"] * m["T"]) * torch.clamp(S[None] - K[:, None], min=0.0).mean(1)
    assert torch.all((p - ref).abs() <= 1e-6 * S.mean()), (p, ref)


@pytest.mark.parametrize("scheme", ["qe", "qem"])
@pytest.mark.parametrize("paths,n_strikes", [(1, 1), (31, 32), (32 * SMS + 1, 1), (32 * SMS * 24 + 5, 33),
                                             (32 * SMS * 150 + 17, 32), (32 * SMS * 40 + 3, 256)])
def test_adjoint_with_a_global_segment_equals_shared_segments(simr, paths, n_strikes, scheme):
    # the two kernels form the same FP32 sums of 32 paths (one hands out items, one
    # strides); an odd step count and one segment past the even one
    K = torch.linspace(80.0, 120.0, n_strikes, dtype=torch.float64, device="cuda") if n_strikes > 1 else \
        torch.tensor([100.0], dtype=torch.float64, device="cuda")
    m = dict(workloads.BASE_MODEL, sigma=0.6)
    with simr.scheme(scheme):
        a = simr.greeks_adjoint(m, K, True, 171, paths, 3)  # 171 steps: one segment, too long for shared memory
        b = simr.greeks_adjoint(m, K, True, 171, paths, 3, ckpt_every=16)
    for x, y in zip(a, b):
        scale = y.abs().amax(dim=0, keepdim=True).clamp_min(1e-300)
        assert torch.all((x - y).abs() <= 1e-11 * scale), float(((x - y).abs() / scale).max())


@pytest.mark.parametrize("scheme", ["qe", "qem"])
@pytest.mark.parametrize("n_assets", [1, 2, 3, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("steps,paths", [(3, 32 * SMS * 17 + 9), (600, 97)])  # 600 steps x 16 assets: no counter table
def test_basket_of_one_weight_is_the_single_asset_price(simr, n_assets, steps, paths, scheme):
    # uncorrelated assets with the last one's weight 1 and the rest 0: the last
    # asset's own European price on the paths of its option index.  FP32 sums of 32
    # paths against 64: 6 roundings of 2^-24 each, 4e-7
    m = workloads.random_models(n_assets, 5)
    for q in m:
        q["T"], q["r"] = 1.0, 0.03
    w = np.zeros(n_assets)
    w[-1] = 1.0
    K = torch.linspace(80.0, 120.0, 33, dtype=torch.float64, device="cuda")
    with simr.scheme(scheme):
        p, _ = simr.basket_price(m, np.eye(n_assets), w, K, False, steps, paths, 7)
        q, _ = simr.price(m[-1], K, False, steps, paths, 7, option_index=n_assets - 1)
    torch.testing.assert_close(p, q, rtol=4e-7, atol=4e-7)


@pytest.mark.parametrize("paths", [2, 63, 65, 64 * SMS * 24 + 1, 64 * SMS * 100 + 31])
@pytest.mark.parametrize("steps", [1, 7, 4095])
def test_one_exercise_date_is_the_european_price(simr, steps, paths):
    # the Longstaff-Schwartz path kernel against the pricing kernel on the same paths
    # (FP32 sums grouped differently: 4e-7 as above, of a mean payoff above 1)
    if steps == 4095 and paths > 70:
        pytest.skip("long paths at small counts only")
    m = dict(workloads.BASE_MODEL)
    p = simr.lsm_price(m, 110.0, True, steps, steps, paths, 5)[0]
    q, _ = simr.price(m, torch.tensor([110.0], dtype=torch.float64, device="cuda"), True, steps, paths, 5)
    torch.testing.assert_close(p, q, rtol=4e-7, atol=4e-7)


def test_book_rows_beyond_one_per_lane(simr):
    # more work items than the reducing warp has lanes, and one path
    book = [dict(model=dict(workloads.BASE_MODEL), K=100.0, is_put=False, steps=3, paths=n) for n in (1, 64 * 33 + 1, 100003)]
    p, se, _ = simr.batch(book, seed=4, autotune=False)
    for i, o in enumerate(book):
        q, sq = simr.price(o["model"], torch.tensor([100.0], dtype=torch.float64, device="cuda"), False, 3, o["paths"], 4,
                           option_index=i)
        torch.testing.assert_close(p[i:i + 1], q, rtol=1e-12, atol=1e-12)
        torch.testing.assert_close(se[i:i + 1], sq, rtol=1e-9, atol=1e-12)
