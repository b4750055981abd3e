"""Which books run account-resident, and that those of test_gpu_acct.py's kinds do: a comparison of the two
forms says something only where each of them ran."""
import dataclasses

import numpy as np
import pytest

from paper_2606_23367_gb300 import build, prism
from paper_2606_23367_gb300.workloads import make_workload
from tests.parity_util import gpu_solve

pytestmark = pytest.mark.gpu
BLOCK, GEMM = (prism.KERNEL_CLASSES.index(k) for k in ("block", "gemm_P"))
BF16, FP32, FP64 = prism.PRISM_BATCHED_BF16, prism.PRISM_BATCHED_FP32, prism.PRISM_PLAIN_FP64


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    prism.load_library()


@pytest.mark.parametrize("N,M", [(2000, 400), (900, 40)])
def test_no_caps_and_infinite_caps_are_the_same_book(N, M):
    # NULL, and an array without a finite cap, in host and in device memory: one route, the same bits
    torch = pytest.importorskip("torch")
    uni, batch = make_workload(1, N=N, K=48, M=M)
    inf = np.full(M, np.inf)
    res = [gpu_solve(uni, dataclasses.replace(batch, turnover_cap=c), precision=BF16)
           for c in (None, inf, torch.as_tensor(inf).cuda())]
    for r in res[1:]:
        assert r["kernel_launches"] == res[0]["kernel_launches"]
        assert np.array_equal(r["w"], res[0]["w"]) and np.array_equal(r["lambda_band"], res[0]["lambda_band"])


def _both_forms(uni, batch, mode, **batched):
    new = gpu_solve(uni, batch, precision=mode)
    old = gpu_solve(uni, batch, precision=mode, **(batched or dict(chains=1)))
    assert new["kernel_launches"][BLOCK] >= 1 and new["kernel_launches"][GEMM] == 0
    assert old["kernel_launches"][GEMM] >= 1 and old["kernel_launches"][BLOCK] == 0
    assert np.array_equal(new["status"], old["status"])
    sure = np.repeat(old["status"] == prism.PRISM_CERTIFIED, np.diff(batch.offsets))
    assert sure.any() and float(np.max(np.abs(new["w"] - old["w"])[sure])) <= 1e-9


# (FP32 rows of 48 factors do not fit eight CTAs at 8,193 names, so that size takes 32 there)
@pytest.mark.parametrize("mode,N,K,S", [(m, *s) for m in (BF16, FP32) for s in
                                        ((160, 1, 20), (256, 16, 20), (257, 17, 20), (1024, 9, 1), (1025, 33, 64), (2048, 8, 20),
                                         (2049, 31, 20), (3000, 64, 20), (8193, 48 if m == BF16 else 32, 20))])
def test_shapes_run_both_forms(mode, N, K, S):
    uni, batch = make_workload(1, N=N, K=K, S=S, M=3, band_hi=0.15 if S == 20 else (np.inf if S == 1 else 0.05))
    _both_forms(uni, batch, mode)


@pytest.mark.parametrize("over", [dict(), dict(lots=False), dict(tau=np.inf), dict(tilt=0.01, bench=True),
                                  dict(factor_bound=(3, 0.03))])
@pytest.mark.parametrize("N", [400, 1500])
def test_lots_cap_tilt_and_factor_bounds_run_both_forms(N, over):
    uni, batch = make_workload(3, N=N, K=20, M=3, **over)
    _both_forms(uni, batch, BF16)


@pytest.mark.parametrize("mode", [BF16, FP32])
@pytest.mark.parametrize("N,K", [(700, 13), (4000, 32)])
def test_ragged_accounts_run_both_forms(mode, N, K):
    uni, batch = make_workload(2, N=N, K=K, M=12)
    _both_forms(uni, batch, mode, ragged_layout=1)
