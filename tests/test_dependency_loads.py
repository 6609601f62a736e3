"""A kernel launched as a programmatic dependent is resident while its
predecessor still writes.  What it reads after its dependency wait must not take
the read-only path (__ldg, const __restrict__ parameters), which is for data that
stays as it is for the kernel's lifetime and whose loads may move above the
wait.  Read from the sources."""
import os
import re

import pytest

from tests.test_cluster_start import CSRC, functions

WAIT = "grid_dependency_wait()"
# a helper of evict_select_kernel, which is launched after its predecessor's end
PLAIN_LAUNCH = {"load4"}


def sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            yield f, open(os.path.join(CSRC, f)).read()


def signature(text, name):
    return re.search(r"\b%s\(((?:[^;{}()]|\([^()]*\))*)\)\s*\{" % name, text).group(1)


FUNCS = [(f, t, n, b) for f, t in sources() for n, b in functions(t)]
DEPENDENT = [(f, t, n, b) for f, t, n, b in FUNCS if WAIT in b]


def test_the_dependent_kernels_are_found():
    assert {n for _, _, n, _ in DEPENDENT} >= {
        "append_kernel", "block_scores_kernel", "compose_kernel", "contrib_mma_kernel",
        "decode_cluster_kernel", "decode_f32_kernel", "decode_merge_kernel", "decode_mma_kernel",
        "decode_radius_kernel", "decode_range_kernel", "decode_reduce_kernel",
        "evict_select_smem_kernel", "gather_rows_kernel", "score_col_f32_kernel",
        "score_col_stream_tc_kernel", "score_col_tc_kernel", "score_lse_f32_kernel",
        "score_lse_tc_kernel", "second_pass_kernel"}


@pytest.mark.parametrize("file,text,name,body", DEPENDENT, ids=[n for _, _, n, _ in DEPENDENT])
def test_no_read_only_loads_after_the_dependency_wait(file, text, name, body):
    assert "__restrict__" not in signature(text, name)
    assert "__ldg(" not in body[body.index(WAIT):]


def test_the_kernels_helpers_take_plain_loads():
    bad = [n for _, t, n, b in FUNCS if "__ldg(" in b and WAIT not in b and n not in PLAIN_LAUNCH and
           "__global__" not in t[max(0, t.index(n + "(") - 120):t.index(n + "(")]]
    assert not bad
