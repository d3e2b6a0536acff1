"""What the kernel of the cell route must do in its source, checked without a GPU: the order of accesses that no run can
be relied on to show."""
import os
import re

import paper_2001_01347_b200.build as build


def kernel_body(name):
    text = open(os.path.join(build.CSRC, "cells.cu")).read()
    text = re.sub(r"//[^\n]*", "", text)
    at = text.index("__global__", text.rindex("\n", 0, re.search(r"\b%s\(" % name, text).start()) - 200)
    start = text.index("{", re.search(r"\b%s\([^)]*\)\s*\{" % name, text[at:]).start() + at)
    depth = 0
    for i in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start:i]
    raise AssertionError("unbalanced braces")


def test_a_cta_writes_to_another_one_only_after_a_cluster_barrier():
    # shared memory of a CTA of the cluster that has not started yet may not be written
    body = kernel_body("k_cells")
    barrier = min(body.index(b) for b in ("barrier_wait()", "cl.sync()") if b in body)
    assert body.index("barrier_arrive()") < body.index("grid_dep_wait()") < barrier
    assert body.index("map_shared_rank") > barrier
