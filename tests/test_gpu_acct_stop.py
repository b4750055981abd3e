"""How accounts of the account-resident iterations stop: the point they stop at, the status they get, and
what a time budget does."""
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
