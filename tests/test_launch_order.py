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
