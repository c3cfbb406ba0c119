"""What bench.py says about the sources: which headers belong to the tiled path alone (an edit there keeps the narrow
kernels' measured traffic), and the FP64 work that the pre-filter still has."""
import os
import re

import bench

CSRC = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_2506_10257_gb300", "csrc")


def reach(*roots):
    seen, todo = set(), list(roots)
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        with open(os.path.join(CSRC, f)) as fh:
            todo += [h for h in re.findall(r'#include "([^"/]+\.cuh)"', fh.read())]
    return seen


def test_tiled_headers_are_those_only_the_tiled_path_includes():
    narrow = reach("rpca_kernels.cuh", "rpca_batch.cuh")
    assert set(bench.TILED_HEADERS) == reach("rpca_wide.cuh") - narrow
    # every header is one or the other
    heads = {f for f in os.listdir(CSRC) if f.endswith(".cuh")}
    assert heads == narrow | set(bench.TILED_HEADERS)


def test_the_prefilter_counts_fp64_work_where_the_kernels_do_it():
    assert bench.prefilter_fp64_ops(87880, 132) == 7 * 87880 * 132
    with open(os.path.join(CSRC, "rpca_prefilter.cu")) as f:
        src = f.read()
    a = src.index("pf_average_kernel(const float*")
    body = src[a:src.index("pf_segment64<HP>(X", a)]
    assert "double" not in body  # its FP64 sums are the rare segments' fallback
