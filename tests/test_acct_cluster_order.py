"""A CTA of a cluster may be reached through distributed shared memory only once it has started: in the
account-resident kernel a barrier over the whole cluster, which nothing but the kernel's cluster form
conditions, stands before the first access to another CTA's shared memory. Read from the source, since a
CTA that starts late cannot be arranged (and must not be tried) on a GPU."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_23367_gb300", "csrc",
                   "acct_admm.cuh")


def test_a_cluster_barrier_comes_before_the_first_remote_access():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    body = text[text.index("k_acct_admm("):]
    remote = body.index("map_shared_rank")
    leave = body.index("return;")                    # an account that does not iterate: the whole cluster leaves
    depth, top = 0, []
    for m in re.finditer(r"[{}]|if constexpr \(CL\) cluster\.sync\(\);", body[:remote]):
        if m.group() in "{}":
            depth += 1 if m.group() == "{" else -1
        elif depth == 1:                             # in the kernel's own scope, under no run-time condition
            top.append(m.start())
    assert top and leave < top[0] < remote
