"""The checkpointed adjoint kernel of one strike: the interval decides between the
variants for five and for four resident blocks, and at 88 steps and more between segments
in shared and in global memory.  The same path whatever the interval, so the same FP32
sums of 32 paths: 1e-11 of the column for the order of their FP64 additions.
"""
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


@pytest.mark.parametrize("scheme", ["qe", "qem"])
@pytest.mark.parametrize("n_strikes", [1, 2])
@pytest.mark.parametrize("steps,paths", [(1, 33), (8, 100003), (95, 40001)])
def test_every_interval_gives_the_same_sums(simr, steps, paths, n_strikes, scheme):
    K = torch.tensor([95.0, 105.0][:n_strikes], dtype=torch.float64, device="cuda")
    m = dict(workloads.BASE_MODEL, sigma=0.9, rho=-0.9, kappa=0.7)
    with simr.scheme(scheme):
        ref = simr.greeks_adjoint(m, K, False, steps, paths, 5, ckpt_every=2)
        for k in (8, 26, 28, 30, 64, 96):
            for x, y in zip(simr.greeks_adjoint(m, K, False, steps, paths, 5, ckpt_every=k), ref):
                scale = y.abs().amax(dim=0, keepdim=True).clamp_min(1e-300)
                assert torch.all((x - y).abs() <= 1e-11 * scale), (k, float(((x - y).abs() / scale).max()))
