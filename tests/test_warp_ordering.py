"""Orderings between lanes that a run cannot show missing (the hardware happens to keep them), read
from the sources."""
import os
import re

from paper_2608_17402_gb300 import _build


def _source(name):
    with open(os.path.join(_build.CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())   # without comments


def _body(src, head):
    """The braces' content that follows the first match of `head`."""
    i = src.index("{", re.search(head, src).end())
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        j += 1
        if depth == 0:
            return src[i:j]


def test_one_lane_wait_publishes_what_it_saw():
    """Lane 0 alone waits on the barrier; another lane may issue what depends on it.  A shuffle
    orders no memory accesses between lanes, __syncwarp does."""
    one = _body(_body(_source("common.cuh"), r"bool mbar_wait_warp\("), r"if \(ONE\)")
    assert re.search(r"__shfl_sync.*__syncwarp\(\)", one, re.S), one


def test_aligned_cluster_barriers_are_reached_converged():
    """barrier.cluster with .aligned wants every lane of the warp to execute it together: directly after
    __syncwarp or __syncthreads, in the function itself or at each of its calls."""
    converged = r"__sync(?:warp|threads)\(\);\s*(?:tc_fence_(?:before|after)\(\);\s*)?$"
    for name in sorted(os.listdir(_build.CSRC)):
        if not name.endswith((".cu", ".cuh", ".h")):
            continue
        src = _source(name)
        for m in re.finditer(r"asm volatile\(\s*\"barrier\.cluster", src):
            before = src[:m.start()]
            if re.search(converged, before):
                continue
            fn = re.findall(r"__device__ __forceinline__ \w+ (\w+)\(", before)[-1]
            calls = [c.start() for c in re.finditer(rf"(?<!void )\b{fn}\(\);", src)]
            assert calls, (name, fn)
            assert all(re.search(converged, src[:c]) for c in calls), (name, fn)
