"""A CTA may touch another CTA's shared memory only once that CTA is known to run. Which barrier
shows it can't be seen from results, so the order is read off the kernels' source (CPU)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1004_0023_gb300", "csrc")


def _function(source, name):
    """The body of the function or kernel definition `name`, without comments."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, source)).read())
    at = re.search(r"\b%s\s*\([^;{]*\)\s*\{" % re.escape(name), text)
    assert at, name
    depth, k = 1, at.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        k += 1
    return text[at.end():k]


# function, the barrier that shows the peers run, the first use of their shared memory
ORDER = [
    ("pt_kernels.cu", "peer_producer", r"cluster_wait_acquire\(\)", r"produce\(0, 0, 0\)"),
    ("pt_kernels.cu", "split_body", r"cluster_barrier\(\)", r"(peer_sp|peer_xch) ?[+\[]|= peer_xch \+"),
    ("pt_kernels.cu", "sweep_classical_kernel", r"cluster_barrier\(\)", r"st_cluster_u64x2\("),
    ("pt_kernels.cu", "sweep_packed_body", r"cluster_barrier\(\)", r"st_cluster_u64x2\("),
    ("pt_kernels.cu", "sweep_packed_body", r"cluster_wait_acquire\(\)", r"map_shared_rank\("),
    ("pt_batch.cu", "run_problem", r"cluster_barrier\(\)", r"st_cluster_u64x2\("),
    ("pt_batch.cu", "batch_kernel", r"cluster\.sync\(\)", r"\*cluster\.map_shared_rank\("),
]


@pytest.mark.parametrize("source,name,barrier,use", ORDER)
def test_peers_are_known_to_run_before_their_shared_memory_is_used(source, name, barrier, use):
    body = _function(source, name)
    shown, first = re.search(barrier, body), re.search(use, body)
    assert shown and first and shown.start() < first.start()


def test_both_ctas_of_a_path_8_cluster_enter_the_barrier_that_the_producer_waits_for():
    """One arrival by every thread before the ranks part, and a wait for it in each before the next
    arrival."""
    kernel = _function("pt_kernels.cu", "sweep_peer_kernel")
    assert kernel.index("cluster_arrive_relaxed()") < kernel.index("block_rank()")
    assert kernel.count("cluster_arrive") == 1 and "cluster_wait" not in kernel
    sweeper = _function("pt_kernels.cu", "sweep_packed_body")
    assert sweeper.index("cluster_wait_acquire()") < sweeper.index("cluster_arrive")
    producer = _function("pt_kernels.cu", "peer_producer")
    assert producer.index("cluster_wait_acquire()") < producer.index("cluster_barrier()")
