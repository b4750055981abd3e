"""The account-resident iterations (every iteration of an account in one launch) against the batched
kernels, which the option chains = 1 keeps a book on: different roundings of the same method, so after
the FP64 polish the same weights (1e-9, the bar of the other pairs of forms). Sizes at the edges of the
kernel's shapes: one and four entries a thread (256 names), 256 and 512 threads (1,024 names), one CTA and
clusters of 2, 4 and 8 (2,048 names, and what fits a CTA's shared memory), factor counts at and off the
16-byte chunks of a row, one sector and the most, sectors smaller than a thread's four entries."""
import dataclasses

import numpy as np
import pytest

from paper_2606_23367_gb300 import build, prism
from paper_2606_23367_gb300.workloads import make_workload
from tests.parity_util import assert_parity, gpu_solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    prism.load_library()


def _agree(uni, batch, mode, **batched):
    new = gpu_solve(uni, batch, precision=mode)
    old = gpu_solve(uni, batch, precision=mode, **(batched or dict(chains=1)))
    assert np.all(new["status"] == old["status"]), (new["status"], old["status"])
    assert np.all(new["status"] == prism.PRISM_CERTIFIED)
    assert float(np.max(np.abs(new["w"] - old["w"]))) <= 1e-9
    return new


@pytest.mark.parametrize("mode", [prism.PRISM_BATCHED_BF16, prism.PRISM_BATCHED_FP32])
@pytest.mark.parametrize("N,K,S", [(160, 1, 20), (256, 16, 20), (257, 17, 20), (1024, 9, 1), (1025, 33, 64), (2048, 8, 20),
                                   (2049, 31, 20), (3000, 64, 20), (8193, 48, 20)])
def test_shapes(mode, N, K, S):
    band = 0.15 if S == 20 else (np.inf if S == 1 else 0.05)
    uni, batch = make_workload(1, N=N, K=K, S=S, M=3, band_hi=band)
    new = _agree(uni, batch, mode)
    if N < 3000:
        assert_parity(uni, batch, new, accounts=[1])


@pytest.mark.parametrize("mode", [prism.PRISM_BATCHED_BF16, prism.PRISM_PLAIN_FP32])
@pytest.mark.parametrize("S,band_hi,floor", [(60, 0.03, 0.012), (20, 0.08, 0.045)])
def test_costs_floors_and_binding_bands(mode, S, band_hi, floor):
    # costs per entry, lower bounds above 0 and band floors and caps that bind, with an upper edge
    # inside a thread's entries. With 60 sectors more bands bind than the polish takes rows (22) for
    # some accounts, which both forms return uncertified
    uni, batch = make_workload(1, N=900, K=24, S=S, M=4, band_hi=band_hi)
    r = np.random.default_rng(3)
    lower = np.where((batch.upper > 0.002) & (r.random(batch.lower.shape) < 0.05), 0.001, 0.0)
    band_lo = np.zeros_like(batch.band_lo)
    band_lo[:, ::7] = floor
    batch = dataclasses.replace(batch, tc=r.uniform(5e-4, 5e-3, size=batch.tc.shape), lower=lower, band_lo=band_lo)
    new = gpu_solve(uni, batch, precision=mode)
    old = gpu_solve(uni, batch, precision=mode, chains=1)
    assert np.any(new["lambda_band"] > 0) and np.any(new["lambda_band"] < 0)
    assert np.all(new["status"] == old["status"])
    assert S == 60 or np.all(new["status"] == prism.PRISM_CERTIFIED)
    assert_parity(uni, batch, new, accounts=np.flatnonzero(new["status"] == prism.PRISM_CERTIFIED))


@pytest.mark.parametrize("over", [dict(), dict(lots=False), dict(tau=np.inf), dict(tilt=0.01, bench=True),
                                  dict(factor_bound=(3, 0.03))])
@pytest.mark.parametrize("N", [400, 1500])
def test_lots_cap_tilt_and_factor_bounds(N, over):
    uni, batch = make_workload(3, N=N, K=20, M=3, **over)
    new = _agree(uni, batch, prism.PRISM_BATCHED_BF16)
    assert_parity(uni, batch, new, accounts=[2])


@pytest.mark.parametrize("N,K", [(700, 13), (4000, 32)])
def test_ragged_accounts_form_their_own_capacitance(N, K):
    # accounts of 100 names up to N, in classes of one CTA and of clusters
    uni, batch = make_workload(2, N=N, K=K, M=12)
    _agree(uni, batch, prism.PRISM_BATCHED_BF16, ragged_layout=1)
    _agree(uni, batch, prism.PRISM_BATCHED_FP32, ragged_layout=1)


@pytest.mark.parametrize("N,K", [(60, 5), (256, 10), (257, 16), (900, 21)])
def test_fp64(N, K):
    uni, batch = make_workload(0, N=N, K=K)
    new = gpu_solve(uni, batch, precision=prism.PRISM_PLAIN_FP64)
    assert_parity(uni, batch, new)


def test_time_budget_stops_every_account():
    # a budget that has run out when the kernel starts: one iteration, no account past it
    uni, batch = make_workload(1, N=900, K=16, M=6)
    res = gpu_solve(uni, batch, precision=prism.PRISM_BATCHED_BF16, time_budget_s=1e-9, polish_rounds=1)
    assert int(res["iters"].max()) == 1
    assert set(res["status"].tolist()) <= {prism.PRISM_TIMEOUT, prism.PRISM_CERTIFIED}
    assert (res["status"] == prism.PRISM_TIMEOUT).any()


@pytest.mark.parametrize("rounds", [None, 3])
@pytest.mark.parametrize("kind,N,M,mode", [(1, 3000, 400, prism.PRISM_BATCHED_BF16), (1, 3000, 400, prism.PRISM_BATCHED_FP32),
                                           (3, 2000, 600, prism.PRISM_BATCHED_BF16)])
def test_a_batched_book_hands_its_last_accounts_over(kind, N, M, mode, rounds):
    # more accounts than the account-resident form is faster for: batched, until few iterate on or few
    # come back from a polish cut short, and the weights of the batched kernels alone
    uni, batch = make_workload(kind, N=N, K=64, S=20, M=M)
    opts = dict(precision=mode, check_every=5, **({} if rounds is None else dict(polish_rounds=rounds)))
    new, old = gpu_solve(uni, batch, **opts), gpu_solve(uni, batch, chains=1, **opts)
    block = prism.KERNEL_CLASSES.index("block")
    assert new["kernel_launches"][block] >= 1 and old["kernel_launches"][block] == 0
    assert new["kernel_launches"][prism.KERNEL_CLASSES.index("gemm_P")] > 0
    sure = old["status"] == prism.PRISM_CERTIFIED
    assert sure.any() and np.all(new["status"][sure] == prism.PRISM_CERTIFIED)
    acct = np.repeat(sure, np.diff(batch.offsets))
    assert float(np.max(np.abs(new["w"] - old["w"])[acct])) <= 1e-9


@pytest.mark.parametrize("mode", [prism.PRISM_BATCHED_BF16, prism.PRISM_BATCHED_FP32])
@pytest.mark.parametrize("seed", [101, 102])
def test_a_band_edge_that_the_bounds_imply_has_no_multiplier(mode, seed):
    # long-only books with band floors of 0: the floor holds by the entries' own bounds, so that its
    # multiplier, which a sector sold out leaves open below 0, is 0
    uni, batch = make_workload(4, seed=seed, N=2000, K=32, M=64, factor_bound=(4, 0.03), tilt=0.01, bench=True)
    assert np.all(batch.lower >= 0) and np.all(batch.band_lo == 0)
    res = gpu_solve(uni, batch, precision=mode)
    assert np.all(res["status"] == prism.PRISM_CERTIFIED)
    assert np.all(res["lambda_band"] >= -1e-12)
