"""A CTA of the tensor-core products that gives up may leave only when no commit of its MMA thread can still arrive at a
barrier in its shared memory: after its loop that thread waits for every barrier that a commit in it
names (wfree, bfree, accfull).  Read off the source; on the way without a failure other warps wait for them too."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_06184_gb300", "csrc")


@pytest.mark.parametrize("name", ["gemm_tc.cu", "gemm_x2.cu"])
def test_every_committed_barrier_is_waited_for(name):
    src = open(os.path.join(CSRC, name)).read()
    role = src[src.index("---------------- MMA issuer"):src.index("---------------- split warps")]
    committed = set(re.findall(r"tc_commit\((\w+)", role))
    waited = set(re.findall(r"mbar_wait\((\w+)", role[role.index("if (last >= 0)"):]))
    assert committed == {"wfree", "bfree", "accfull"} and committed <= waited, (committed, waited)
