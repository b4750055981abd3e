"""The setup that runs on the device: the universe's B gathered, checked and converted there, and a book's
bands and caps checked by the launch that converts them, from host and from device buffers alike. The
same arithmetic on the same values, so the same bits; what is not finite or not ordered is refused."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2606_23367_gb300 import build, prism
from paper_2606_23367_gb300.workloads import make_workload
from tests.parity_util import gpu_solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    prism.load_library()


def _on_device(obj, names):
    return dataclasses.replace(obj, **{n: torch.as_tensor(getattr(obj, n)).cuda() for n in names if getattr(obj, n) is not None})


@pytest.mark.parametrize("N,K,S", [(40, 1, 1), (129, 7, 5), (1000, 64, 64)])
def test_host_and_device_buffers_give_the_same_bits(N, K, S):
    uni, batch = make_workload(1, N=N, K=K, S=S, M=3, band_hi=np.inf)
    batch = dataclasses.replace(batch, upper=np.ones_like(batch.upper))
    a = gpu_solve(uni, batch, precision=prism.PRISM_BATCHED_BF16)
    dev_uni = _on_device(uni, ("B", "f", "d", "mu", "sector"))
    dev_batch = _on_device(batch, ("w0", "lower", "upper", "tc", "band_lo", "band_hi"))
    b = gpu_solve(dev_uni, dev_batch, precision=prism.PRISM_BATCHED_BF16)
    for k in ("w", "status", "iters", "nu", "lambda_band"):
        x, y = (np.asarray(v.cpu() if hasattr(v, "cpu") else v) for v in (a[k], b[k]))
        assert np.array_equal(x, y), k
    assert np.all(np.asarray(a["status"]) == prism.PRISM_CERTIFIED)


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("at", [(0, 0), (299, 12)])
def test_a_value_of_B_that_is_not_finite_is_refused(device, value, at):
    uni, _ = make_workload(1, N=300, K=13, M=1)
    B = uni.B.copy()
    B[at] = value
    uni = dataclasses.replace(uni, B=B)
    if device:
        uni = _on_device(uni, ("B",))
    with pytest.raises(prism.PrismError) as ei:
        prism.create_universe(uni)
    assert ei.value.code == prism.PRISM_ERR_ARGUMENT


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("field,value", [("band_lo", np.nan), ("band_hi", np.nan), ("band_lo", np.inf), ("turnover_cap", np.nan),
                                         ("turnover_cap", -1e-9)])
def test_bands_and_caps_out_of_order_are_refused(device, field, value):
    uni, batch = make_workload(1, N=300, K=8, M=4)
    x = np.full(4, np.inf) if field == "turnover_cap" else np.array(getattr(batch, field), copy=True)
    x.reshape(-1)[-1] = value                          # the last account's, the last sector's
    batch = dataclasses.replace(batch, **{field: x})
    if device:
        batch = _on_device(batch, (field,))
    with pytest.raises(prism.PrismError) as ei:
        gpu_solve(uni, batch, precision=prism.PRISM_BATCHED_FP32)
    assert ei.value.code == prism.PRISM_ERR_ARGUMENT


def test_a_rejected_account_returns_zeros_beside_others():
    uni, batch = make_workload(1, N=600, K=16, M=3)
    sl = batch.account_slice(1)
    batch.upper[sl] = 1e-4                             # capacity far below the budget
    first = gpu_solve(uni, batch, precision=prism.PRISM_BATCHED_BF16)
    assert first["status"].tolist() == [prism.PRISM_CERTIFIED, prism.PRISM_NO_FEASIBLE_RETURN, prism.PRISM_CERTIFIED]
    assert not np.any(first["w"][sl])


@pytest.mark.parametrize("device", [False, True])
def test_a_universe_holds_its_arrays_and_no_scratch(device):
    N, K = 100_000, 64
    uni, _ = make_workload(1, N=N, K=K, M=1)
    if device:
        uni = _on_device(uni, ("B",))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h = prism.create_universe(uni)
    held = before - torch.cuda.mem_get_info()[0]
    h.close()
    # B in FP64, FP32 and BF16, and padded and transposed copies of the last two; per asset some 40 bytes of the
    # model and the order; per penalty six matrices in FP32; blocks of 2 MB
    want = N * (8 * K + 2 * 4 * K + 4 * 2 * K + 40) + 33 * 6 * 4 * K * K
    assert held <= want + (4 << 20), (held, want)
