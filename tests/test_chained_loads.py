"""Loads of kernels that are set up while the kernel before them still runs.

Such a kernel (its first act is chain_wait) may hold a place on an SM while
its predecessor writes, so nothing that a kernel of the library writes is
read-only for its lifetime, which is what the read-only path (__ldg, and
const __restrict__ parameters, which the compiler may load through it) asks
for.  A stale word there would be a race on memory, so this is checked by
reading the sources and not on a GPU."""
import glob
import os
import re

import pytest

from paper_2205_11048_gb300 import build as BLD

# arrays that only the host writes, while no kernel runs: the decay weights
HOST_WRITTEN = ("a.wtab",)
FILES = sorted(glob.glob(os.path.join(BLD.CSRC, "*.cu")) +
               glob.glob(os.path.join(BLD.CSRC, "*.cuh")))


def code_of(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def kernels(code):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s*(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?"
                         r"(\w+)\(([^{;]*)\)\s*\{", code):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            i += 1
        yield m.group(1), m.group(2), code[m.end():i]


def test_the_chained_kernels_are_found():
    found = {name for p in FILES for name, _, body in kernels(code_of(p)) if "chain_wait()" in body}
    assert found == {"k_message_weights", "k_sort_histogram", "k_onesweep", "k_seg_scan",
                     "k_row_apply", "k_row_long", "k_pull_rows", "k_push_copy", "k_dense_accumulate"}
    launched = {m for p in FILES for m in re.findall(r"launch_chained\([^;]*?\b(k_\w+)", code_of(p))}
    assert launched <= found


@pytest.mark.parametrize("path", FILES, ids=[os.path.basename(p) for p in FILES])
def test_chained_kernels_do_not_use_the_read_only_path(path):
    code = code_of(path)
    for name, params, body in kernels(code):
        if "chain_wait()" in body:
            bad = [p.strip() for p in params.split(",") if "const" in p and "__restrict__" in p]
            assert not bad, (name, bad)
    args = re.findall(r"__ldg\(\s*([^;]*)", code) + re.findall(r"(ld\.global\.nc[^;]*)", code)
    assert [a for a in args if not a.startswith(HOST_WRITTEN)] == []
