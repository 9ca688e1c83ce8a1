"""Kernels may become resident while the kernel before them still runs (programmatic dependent launch), and that kernel may be
the caller's own, for instance the one that advances kv_len: a kernel's first look at memory must come behind its wait."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_18753_b200", "csrc")


def _kernels():
    """(file, name, body without comments) of every __global__ function that waits for its predecessor."""
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for part in re.split(r"__global__", text)[1:]:
            kernel = re.search(r"(\w+_kernel)\s*\(", part)
            body = part[part.index("{"):]
            if kernel and "chain_wait()" in body:
                yield name, kernel.group(1), body


def test_there_are_kernels_to_look_at():
    names = {k for _, k, _ in _kernels()}
    assert {"decode_sm100_kernel", "decode_select_kernel", "decode_scores_kernel", "decode_route_kernel", "summaries_kernel"} <= names


@pytest.mark.parametrize("name,kernel,body", list(_kernels()), ids=lambda v: v if len(v) < 40 else "")
def test_caller_arrays_are_read_behind_the_wait(name, kernel, body):
    before = body[:body.index("chain_wait()")]
    # a lambda that is only defined before the wait, and called behind it, reads nothing there
    before = re.sub(r"auto \w+ = \[&\]\([^)]*\) \{(?:[^\n]*\};|[^\n]*\n.*?\n  \};)", "", before, flags=re.S)
    assert not re.search(r"(kv_len|count|blk_idx|blk_bias|mask|page_table|Kbar)\s*\[|__ld\w*\(|sequence_length\(", before), (name, kernel)
