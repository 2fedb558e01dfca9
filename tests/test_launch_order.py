"""Orders between kernels that only the sources can show without running a race: which wait
stands before which signal."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_24793_gb300", "csrc")


def _code(name: str) -> str:
    """The source without its // comments."""
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("name", ["verify_attn.cu", "verify_attn_tcq.cu", "verify_attn_tcq2.cu", "verify_attn_tcp.cu"])
def test_attention_lets_dependents_start_only_after_its_own_wait(name):
    """A launch under the stable-cache promise reads the cache as soon as it starts, so a launch
    without the promise may let it start only once everything before (a commit two launches
    back) is done."""
    code = _code(name)
    waits = [m.start() for m in re.finditer(r"if \(!p\.kv_stable\) griddep_wait\(\);", code)]
    signals = [m.start() for m in re.finditer(r"griddep_launch_dependents\(\);", code)]
    assert len(waits) == len(signals) == 1
    assert waits[0] < signals[0]


def test_lmhead_pair_leaves_after_the_last_signal_of_its_mmas():
    """The leader's commits signal barriers in both CTAs of a pair: both wait for the last one,
    before the cluster barrier that lets them leave."""
    code = _code("lmhead.cu")
    assert re.search(r"umma_commit_pair_on\(on, mma_done, 3\);", code)
    waits = [m.start() for m in re.finditer(r"mbar_wait\(mma_done, 0, WAIT_NS\)", code)]
    assert len(waits) == 1
    # outside the roles (a role's own code is inside if (rank == 0)), between the block's and the cluster's barrier
    tail = code[code.index("tmem_dealloc_pair") - 900:code.index("tmem_dealloc_pair")]
    order = [tail.index(x) for x in ("__syncthreads();", "if (warp == 1) mbar_wait(mma_done", "cluster_arrive();", "cluster_wait();")]
    assert order == sorted(order)
