"""Kernels that may start before the one ahead of them has finished promise
nothing about the memory they read: no __restrict__ on their pointers and no
read-only loads, under which a load may be moved above the wait, in the kernels
that wait or in the headers whose device code they run."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1702_07961_gb300", "csrc")
PROMISE = re.compile(r"__restrict__|__ldg\s*\(|ld\.global\.nc")


def text(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def closing(s, at, pair):
    """Index past the bracket that closes the first one of `pair` at or after `at`."""
    depth, i = 0, s.index(pair[0], at)
    while True:
        depth += (s[i] == pair[0]) - (s[i] == pair[1])
        i += 1
        if depth == 0:
            return i


def kernels(s):
    for m in re.finditer(r"__global__", s):
        name = re.compile(r"\b(\w+_kernel)\s*\(").search(s, m.start())
        params = closing(s, name.end() - 1, "()")
        yield name.group(1), s[name.start():closing(s, params, "{}")]


WAITING = [(os.path.basename(p), k, body) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))
           for k, body in kernels(text(p)) if "griddep_wait()" in body]


def test_the_kernels_are_found():
    assert {k for _, k, _ in WAITING} >= {"tile_sort_kernel", "tile_sort_composite_kernel", "splitter_kernel",
                                          "merge_pass_kernel", "merge_pipelined_kernel", "seg_plan_kernel",
                                          "seg_scan_kernel", "seg_desc_kernel", "seg_merge_kernel"}


@pytest.mark.parametrize("file,kernel,body", WAITING, ids=[k for _, k, _ in WAITING])
def test_a_waiting_kernel_promises_nothing(file, kernel, body):
    assert not PROMISE.search(body), f"{file}: {kernel}"


@pytest.mark.parametrize("header", ["tile_sort.cuh", "splitter.cuh", "merge_tile.cuh", "mms_common.cuh"])
def test_the_shared_device_code_promises_nothing(header):
    assert not PROMISE.search(text(os.path.join(CSRC, header)))


def test_the_descriptor_load_promises_nothing():
    s = text(os.path.join(CSRC, "segmented.cu"))
    assert not PROMISE.search(s)
