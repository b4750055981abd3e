"""How accounts of the account-resident iterations stop: the point they stop at, the status they get, and
what a time budget does."""
import dataclasses

import numpy as np
import pytest

from paper_2606_23367_gb300 import build, prism
from paper_2606_23367_gb300.workloads import make_workload
from tests.parity_util import gpu_solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    prism.load_library()


@pytest.mark.parametrize("max_iter", [2, 3, 5])
@pytest.mark.parametrize("mode,N,K,tol", [(prism.PRISM_BATCHED_BF16, 900, 16, 1e-6), (prism.PRISM_BATCHED_FP32, 900, 16, 1e-6),
                                          (prism.PRISM_BATCHED_BF16, 3000, 64, 1e-6), (prism.PRISM_PLAIN_FP64, 300, 10, 1e-13)])
def test_the_point_an_account_stops_at_meets_its_budget(mode, N, K, tol, max_iter):
    # an account that does not certify is returned as its iterations stop: the budget's root is at its
    # tolerance there, in FP32 beside the rounding of a sum to 1 over at most 32 levels; in FP64 the weights
    # are stored in FP32
    uni, batch = make_workload(1, N=N, K=K, M=6)
    res = gpu_solve(uni, batch, precision=mode, max_iter=max_iter, polish_rounds=1)
    left = res["status"] != prism.PRISM_CERTIFIED
    assert left.any()
    rounding = 32 * 2.0**-24 if mode != prism.PRISM_PLAIN_FP64 else 2.0**-24
    assert float(np.max(res["diag"][left, prism.PRISM_DIAG_BUDGET])) <= tol + rounding


def test_an_account_that_met_its_target_is_not_timed_out():
    # under a cap an account goes on past its target until its entries settle: the iteration cap ends that wait
    # and is no timeout. With 60 sectors more bands bind than the polish takes rows (22) for one account, so
    # that its status comes from the iterations; min_iter puts the target's iteration (40) below the cap (45)
    uni, batch = make_workload(1, N=900, K=24, S=60, M=4, band_hi=0.03)
    r = np.random.default_rng(3)
    lower = np.where((batch.upper > 0.002) & (r.random(batch.lower.shape) < 0.05), 0.001, 0.0)
    band_lo = np.zeros_like(batch.band_lo)
    band_lo[:, ::7] = 0.012
    batch = dataclasses.replace(batch, tc=r.uniform(5e-4, 5e-3, size=batch.tc.shape), lower=lower, band_lo=band_lo,
                                turnover_cap=np.full(4, 5.0))
    opts = dict(precision=prism.PRISM_BATCHED_BF16, min_iter=40, max_iter=15, eps_admm=0.1, eps_kkt=1e-4)
    new, old = gpu_solve(uni, batch, **opts), gpu_solve(uni, batch, chains=1, **opts)
    assert old["status"].tolist().count(prism.PRISM_FEASIBLE_NONCERTIFIED) == 1
    assert np.array_equal(new["status"], old["status"])


def test_fp64_accounts_run_through_a_time_budget():
    # PLAIN_FP64 looks at the budget between accounts, not within one
    uni, batch = make_workload(1, N=300, K=10, M=4)
    res = [gpu_solve(uni, batch, precision=prism.PRISM_PLAIN_FP64, time_budget_s=t) for t in (0.0, 1e-9)]
    assert np.array_equal(res[0]["iters"], res[1]["iters"]) and np.array_equal(res[0]["w"], res[1]["w"])
    assert np.all(res[1]["status"] == prism.PRISM_CERTIFIED)


@pytest.mark.parametrize("shift", [64.0, 1024.0, 8192.0])
def test_a_tilt_that_cancels_mu_is_certified_on_exact_conditions(shift):
    # mu + shift and a tilt of -shift: the same problem, whose FP32 sum is off by the rounding of the large
    # terms. A certified account has the weights of the book without the shift (FP64 rounds mu + shift to
    # 2^-53 x 8192 = 9e-13, at a curvature of 0.01 or more)
    uni, batch = make_workload(4, N=900, K=16, M=16)
    base = gpu_solve(uni, batch, precision=prism.PRISM_BATCHED_BF16)
    assert np.all(base["status"] == prism.PRISM_CERTIFIED)
    uni2 = dataclasses.replace(uni, mu=uni.mu + shift)
    res = gpu_solve(uni2, dataclasses.replace(batch, mu_tilt=np.full(len(batch.w0), -shift)),
                    precision=prism.PRISM_BATCHED_BF16, max_iter=30, polish_rounds=60)
    assert np.mean(res["status"] == prism.PRISM_CERTIFIED) >= 0.5
    sure = np.repeat(res["status"] == prism.PRISM_CERTIFIED, np.diff(batch.offsets))
    assert float(np.max(np.abs(res["w"] - base["w"])[sure])) <= 1e-9


def test_debug_counters_are_those_of_the_call(monkeypatch, capfd):
    # on a handle whose last call counted the batched kernels' root evaluations
    monkeypatch.setenv("PRISM_DEBUG_STATS", "1")
    uni, batch = make_workload(1, N=900, K=16, M=6)
    h = prism.create_universe(uni)
    try:
        for opts in (dict(chains=1), {}):
            capfd.readouterr()
            prism.solve(h, batch, precision=prism.PRISM_BATCHED_BF16, **opts)
            err = capfd.readouterr().err
            assert ("prox account-calls 0," in err) == (not opts), err
    finally:
        h.close()
