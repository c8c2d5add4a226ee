"""commit_load may run before its kernel's dependency wait, while other SMs'
writes of the step before are newer than what this SM's L1 holds: every read of
the state in it has to bypass L1."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2608_22646_gb300", "csrc", "commit.cuh")


def test_commit_load_reads_bypass_l1():
    src = open(SRC).read()
    body = src[src.index("void commit_load("):]
    body = body[:body.index("\n}\n")]
    reads = re.findall(r"(__ldcg\(&)?p\.(st\.\w+|row_of)\[", body)
    assert len(reads) == 8
    assert [name for cached, name in reads if not cached] == []
