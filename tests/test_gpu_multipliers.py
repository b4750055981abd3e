"""The multipliers of the account-resident iterations against those of the batched kernels (chains = 1).
Where a band's multiplier is not unique (a floor of 0 on a sector sold out, which its entries' bounds
imply), the polish keeps the one that its start leads to, 0 or that of the bounds; so the two forms have to
be the same splitting with the same penalties, not only agree in the weights. The seeds hold such accounts.
Tolerance: both forms end in the same FP64 polish, whose multipliers are exact to some 1e-15 of values below 1."""
import numpy as np
import pytest

from paper_2606_23367_gb300 import build, prism
from paper_2606_23367_gb300.workloads import make_workload
from tests.parity_util import gpu_solve

pytestmark = pytest.mark.gpu
BLOCK = prism.KERNEL_CLASSES.index("block")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    prism.load_library()


def _same(uni, batch, mode, **batched):
    new = gpu_solve(uni, batch, precision=mode)
    old = gpu_solve(uni, batch, precision=mode, **batched)
    assert new["kernel_launches"][BLOCK] > 0 and old["kernel_launches"][BLOCK] == 0
    assert np.array_equal(new["status"], old["status"]) and np.all(old["status"] == prism.PRISM_CERTIFIED)
    for k in ("w", "nu", "lambda_band", "theta", "kappa"):
        assert float(np.max(np.abs(new[k] - old[k]))) <= 1e-11, k
    return new


@pytest.mark.parametrize("seed", [5, 39])
def test_a_small_book(seed):
    uni, batch = make_workload(1, seed=seed, N=777, K=17, M=37)
    new = _same(uni, batch, prism.PRISM_BATCHED_BF16, chains=1)
    assert np.any(new["lambda_band"] < -1e-9)          # (an account that keeps the bounds' multiplier)


@pytest.mark.parametrize("seed", [5, 13, 101])
def test_a_mandate_with_benchmark_tilt_and_factor_bounds(seed):
    uni, batch = make_workload(4, seed=seed, N=2000, K=32, M=64, factor_bound=(4, 0.03), tilt=0.01, bench=True)
    _same(uni, batch, prism.PRISM_BATCHED_BF16, chains=1)


@pytest.mark.parametrize("seed", [6, 29, 30, 33, 45, 115])
def test_ragged_accounts(seed):
    # accounts of 100 names up to the universe: iterated over all its positions in either form
    uni, batch = make_workload(2, seed=seed, N=1500, K=24, M=128)
    _same(uni, batch, prism.PRISM_BATCHED_BF16, ragged_layout=1)


@pytest.mark.parametrize("layout", [0, 1, 2])
def test_diagnostics_of_ragged_accounts_that_do_not_certify(layout):
    # on a handle that has held another book of the same shape: nothing of it may reach an account's
    # diagnostics, which are those of the weights returned, nor a gradient
    uni, batch = make_workload(2, seed=3, N=1500, K=24, M=64)
    _, other = make_workload(2, seed=4, N=1500, K=24, M=64)
    h = prism.create_universe(uni)
    try:
        for b in (batch, other):                       # (the workspace has its size after the first two)
            prism.solve(h, b, precision=prism.PRISM_BATCHED_BF16, ragged_layout=layout)
        res = prism.solve(h, batch, precision=prism.PRISM_BATCHED_BF16, ragged_layout=layout, max_iter=2, polish_rounds=1,
                          keep_for_backward=1)
        left = np.flatnonzero(res["status"] != prism.PRISM_CERTIFIED)
        assert len(left) > 0 and not np.any(res["status"] == prism.PRISM_NUMERICAL_FAILURE)
        for a in left:
            sl = batch.account_slice(a)
            w, i = res["w"][sl], batch.asset_idx[sl]
            h_ = uni.B[i].T @ w
            sums = np.bincount(uni.sector[i], w, uni.n_sectors)
            obj = h_ @ (uni.f * h_) + w @ (uni.d[i] * w) - uni.mu[i] @ w + np.abs(w - batch.w0[sl]) @ batch.tc[sl]
            want = {prism.PRISM_DIAG_BUDGET: abs(w.sum() - 1.0), prism.PRISM_DIAG_OBJ: obj,
                    prism.PRISM_DIAG_EXPOSURE: max(0.0, np.max(sums - batch.band_hi[a]), np.max(batch.band_lo[a] - sums))}
            for col, v in want.items():
                assert abs(res["diag"][a, col] - v) <= 1e-12, (a, col)
        grad = prism.prism_solve_batch_backward(res["state"], np.ones(len(batch.w0)))
        assert all(np.all(np.isfinite(grad[k])) for k in ("dmu", "dB", "dd", "dw0"))
        res["state"].close()
    finally:
        h.close()


@pytest.mark.parametrize("seed", [13, 0])
def test_fp64_iterations_are_those_of_the_blocks(seed):
    # the same penalties in FP64, so the same iterates up to rounding: they stop at the same iteration, or at the
    # next where a residual sits on the target
    uni, batch = make_workload(1, seed=seed, N=777, K=17, M=37)
    new = gpu_solve(uni, batch, precision=prism.PRISM_PLAIN_FP64)
    old = gpu_solve(uni, batch, precision=prism.PRISM_PLAIN_FP64, chains=1)
    assert np.array_equal(new["status"], old["status"]) and np.all(old["status"] == prism.PRISM_CERTIFIED)
    assert int(np.max(np.abs(new["iters"] - old["iters"]))) <= 1
    for k in ("w", "nu", "lambda_band"):
        assert float(np.max(np.abs(new[k] - old[k]))) <= 1e-11, k


@pytest.mark.parametrize("seed,N,K,M", [(1160, 492, 39, 162), (1023, 674, 21, 19), (37, 1924, 48, 200)])
def test_lots_and_a_cap_certify_the_same_accounts(seed, N, K, M):
    # books with an account that the polish leaves at first: it certifies where the batched kernels' does, and
    # where it does not, its last polish started from the same iterate and left the same multipliers
    uni, batch = make_workload(3, seed=seed, N=N, K=K, M=M)
    new = gpu_solve(uni, batch, precision=prism.PRISM_BATCHED_BF16)
    old = gpu_solve(uni, batch, precision=prism.PRISM_BATCHED_BF16, chains=1)
    sure = old["status"] == prism.PRISM_CERTIFIED
    assert new["kernel_launches"][BLOCK] > 0 and np.array_equal(new["status"] == prism.PRISM_CERTIFIED, sure)
    for k in ("nu", "lambda_band", "theta"):
        assert float(np.max(np.abs(new[k] - old[k]))) <= 1e-11, k
    assert float(np.max(np.abs(new["w"] - old["w"])[np.repeat(sure, np.diff(batch.offsets))])) <= 1e-11
