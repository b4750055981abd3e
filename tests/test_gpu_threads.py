"""Threads with a universe each: the limits that a launch sets belong to the process, so that accounts and
universes of other sizes in another thread must not lower them in between."""
import threading

import numpy as np
import pytest

from paper_2606_23367_gb300 import build, prism
from paper_2606_23367_gb300.workloads import make_workload

pytestmark = pytest.mark.gpu


def test_threads_with_accounts_of_other_sizes():
    build.build()
    prism.load_library()
    sizes = [(300, 4), (700, 60)] * 4                 # some 20 and 200 KB of shared memory in the same kernel
    made = [make_workload(1, N=N, K=K, M=1) for N, K in sizes]
    handles = [prism.create_universe(u) for u, _ in made]
    want = [prism.solve(h, b, precision=prism.PRISM_BATCHED_FP32) for h, (_, b) in zip(handles, made)]
    gate, wrong = threading.Barrier(len(sizes)), []

    def work(h, b, r):
        gate.wait()
        for _ in range(200):
            try:
                if not np.array_equal(prism.solve(h, b, precision=prism.PRISM_BATCHED_FP32)["w"], r["w"]):
                    wrong.append("other weights")
            except prism.PrismError as e:
                wrong.append(str(e))

    def create(u):
        gate2.wait()
        for _ in range(400):
            try:
                prism.create_universe(u).close()
            except prism.PrismError as e:
                wrong.append(str(e))

    threads = [threading.Thread(target=work, args=(h, b, r)) for h, (_, b), r in zip(handles, made, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    gate2 = threading.Barrier(len(sizes))
    threads = [threading.Thread(target=create, args=(u,)) for u, _ in made]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for h in handles:
        h.close()
    assert not wrong, (len(wrong), wrong[:3])
