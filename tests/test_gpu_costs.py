"""The cost rows of tax lots and the tilts, built on the device: what was refused stays refused with the
same code, and lots at the edges of their cases (harvested lots, a lot of size zero, holdings outside the
box, names whose box is a point, four equal lots) give the oracle's weights."""
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


def _set(arr, at, value):
    out = arr.copy()
    out[at] = value
    return out


@pytest.mark.parametrize("what,code", [
    ("offsets", prism.PRISM_ERR_ARGUMENT), ("count", prism.PRISM_ERR_UNSUPPORTED), ("lower", prism.PRISM_ERR_ARGUMENT),
    ("size", prism.PRISM_ERR_ARGUMENT), ("kappa", prism.PRISM_ERR_ARGUMENT), ("sum", prism.PRISM_ERR_ARGUMENT),
    ("tilt", prism.PRISM_ERR_ARGUMENT), ("bench", prism.PRISM_ERR_ARGUMENT)])
def test_refused(what, code):
    uni, b = make_workload(3, N=400, K=12, M=2, tilt=0.01, bench=True)
    e = int(np.flatnonzero(np.diff(b.lot_offsets) >= 2)[0])        # an entry with two lots or more
    l0 = int(b.lot_offsets[e])
    if what == "offsets":
        b = dataclasses.replace(b, lot_offsets=_set(b.lot_offsets, e + 1, l0 - 1))
    elif what == "count":
        extra = b.lot_offsets.copy()
        extra[e + 1:] += 4
        b = dataclasses.replace(b, lot_offsets=extra, lot_size=np.insert(b.lot_size, l0, np.zeros(4)),
                                lot_kappa=np.insert(b.lot_kappa, l0, np.zeros(4)))
    elif what == "lower":
        b = dataclasses.replace(b, lower=_set(b.lower, e, -0.1))
    elif what == "size":
        b = dataclasses.replace(b, lot_size=_set(b.lot_size, l0, -0.1))
    elif what == "kappa":
        b = dataclasses.replace(b, lot_kappa=_set(b.lot_kappa, l0, np.nan))
    elif what == "sum":
        b = dataclasses.replace(b, lot_size=_set(b.lot_size, l0, b.lot_size[l0] + 0.01))
    elif what == "tilt":
        b = dataclasses.replace(b, mu_tilt=_set(b.mu_tilt, 5, np.inf))
    else:
        b = dataclasses.replace(b, w_bench=_set(b.w_bench, 5, np.nan))
    with pytest.raises(prism.PrismError) as ei:
        gpu_solve(uni, b, precision=prism.PRISM_BATCHED_BF16)
    assert ei.value.code == code


@pytest.mark.parametrize("opts", [{}, {"chains": 1}])
@pytest.mark.parametrize("tilt", [0.0, 0.01])
def test_edges_of_lots(opts, tilt):
    uni, b = make_workload(3, N=400, K=12, M=3, restrict=0.0, tilt=tilt)
    held = np.flatnonzero((np.diff(b.lot_offsets) > 0) & (b.w0 < 0.008))
    size, kappa, upper = b.lot_size.copy(), b.lot_kappa.copy(), b.upper.copy()
    for j, e in enumerate(held[:60]):
        l = slice(int(b.lot_offsets[e]), int(b.lot_offsets[e + 1]))
        n = l.stop - l.start
        if j % 5 == 0:
            kappa[l] = -0.02                                       # harvested: 2 c + kappa < 0
        elif j % 5 == 1:
            kappa[l] = 0.03                                        # equal lots
        elif j % 5 == 2 and n > 1:
            size[l] = 0.0                                          # all in the first lot
            size[l.start] = b.w0[e]
        elif j % 5 == 3:
            upper[e] = 0.5 * b.w0[e]                               # more held than allowed
        else:
            upper[e] = 0.0                                         # a point
    b = dataclasses.replace(b, lot_size=size, lot_kappa=kappa, upper=upper, turnover_cap=np.full(3, 0.6))
    assert_parity(uni, b, gpu_solve(uni, b, precision=prism.PRISM_BATCHED_BF16, **opts))
