"""A CTA may access another CTA's shared memory only once that CTA has started:
every function that maps such an address (`cluster_map`) has waited on a cluster
barrier before.  Read from the sources: the mistake needs no GPU to show, and on
one it would be a race."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_21475_gb300", "csrc")
WAITS = ("cluster_barrier()", "cluster_wait_acquire()")


def functions(text):
    """(name, body) of every function defined at the outer level of a source file."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"^[_a-zA-Z][^;{}#]*?(\w+)\((?:[^;{}()]|\([^()]*\))*\)\s*\{", text, re.M):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


CASES = [(f, name, body) for f in sorted(os.listdir(CSRC)) if f.endswith(".cu")
         for name, body in functions(open(os.path.join(CSRC, f)).read()) if "cluster_map(" in body]


def test_the_kernels_that_share_across_ctas_are_found():
    assert {n for _, n, _ in CASES} >= {"decode_cluster_kernel", "score_lse_f32_kernel",
                                        "score_lse_tc_kernel", "choose_digit", "cluster_scan",
                                        "evict_select_smem_kernel"}


@pytest.mark.parametrize("file,name,body", CASES, ids=[f"{f}:{n}" for f, n, _ in CASES])
def test_a_cluster_barrier_comes_before_the_first_remote_access(file, name, body):
    before = body[:body.index("cluster_map(")]
    assert any(w in before for w in WAITS)
