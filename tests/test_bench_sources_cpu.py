"""The benchmark's traffic figure is tied to the sources of the kernel it was
measured on: all of them, the summary names that kernel, and the operation count
of the N = 4096 tensor-core form."""
import os
import re

import bench


def included(path, seen):
    """`path` and every file of the library that it includes, directly or not."""
    seen.add(path)
    for name in re.findall(r'#include "([^"]+)"', open(os.path.join(bench.ROOT, path)).read()):
        child = os.path.join(os.path.dirname(path), name)
        if child not in seen and os.path.exists(os.path.join(bench.ROOT, child)):
            included(child, seen)
    return seen


def test_every_source_of_the_kernel_is_hashed():
    assert set(bench.KERNEL_SOURCES) == included("paper_1910_01972_gb300/csrc/ols_forward.cu", set())


def test_summary_names_the_kernel():
    kernel = re.search(r"kernel: `(\w+)", open(bench.TRAFFIC_FILE).read()).group(1)
    assert any(re.search(r"\b%s\b" % kernel, open(os.path.join(bench.ROOT, p)).read()) for p in bench.KERNEL_SOURCES)


def test_tensor_operations_at_4096():
    # two radix-64 stages x three split products x eight K steps of 16 per pair of segments
    assert bench.tc64_flops(64, 4680) == 2340 * 65 * 2 * 3 * 8 * (2 * 128 * 128 * 16)
    assert bench.tc64_flops(1, 3) == 2 * 2 * 2 * 3 * 8 * (2 * 128 * 128 * 16)     # an idle half tile counts
