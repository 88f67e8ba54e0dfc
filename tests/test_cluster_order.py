"""Kernels whose CTAs write into one another's shared memory (map_shared_rank): a CTA
may not touch another's shared memory before that one has started, and what a CTA
sets up in its own arrays has to be there before another writes into them.  So a
cluster-wide barrier, or an arrival and its wait, stands before the first such
write, and the arrival after the set-up.  Read from the source: a run shows such a
fault only when a CTA starts late, and then as a wrong address.  No GPU involved."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1712_08872_gb300", "csrc")


def kernel_body(source, name):
    with open(os.path.join(CSRC, source)) as fh:
        text = re.sub(r"//[^\n]*", "", fh.read())
    at = text.index("{", text.index(name + "("))
    depth = 0
    for end in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        if depth == 0:
            return text[at:end]
    raise AssertionError("unbalanced braces")


# (kernel, what a CTA sets in its own shared memory that others write into)
@pytest.mark.parametrize("source,name,setup", [
    ("acr_setup_kernels.cu", "k_leaf_inv_d", "step[tid] = -1;"),
    ("acr_setup_kernels.cu", "k_leaf_inv_f", None),
    ("acr_core_kernels.cu", "void orth", None)])
def test_cluster_has_started_before_the_first_remote_write(source, name, setup):
    body = kernel_body(source, name)
    remote = body.index("map_shared_rank")
    sync, arrive, wait = (body.find(c) for c in ("cl.sync()", "cl.barrier_arrive()",
                                                 "cl.barrier_wait()"))
    if 0 <= sync < remote:
        first = sync
    else:
        assert 0 <= arrive < wait < remote, "no cluster barrier before the first remote write"
        first = arrive
    if setup:
        assert 0 <= body.find(setup) < first, "own arrays are set after the arrival"
