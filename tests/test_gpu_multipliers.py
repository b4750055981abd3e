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
