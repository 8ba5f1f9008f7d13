"""Kernels that start before the kernel ahead of them has ended (launch_after,
grid_begin) must not read what that kernel wrote through the read-only path:
it is for data that nobody writes while the grid exists.  Checked on the
source of the kernels' loads."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_25453_gb300", "csrc")
# written by a kernel of the same call: row and column maxima, sums of squares, digit sums, exponents,
# int32 and residue planes
PRODUCED = ("maxbits", "acc", "sumA", "sumB", "EA", "FB", "Cs", "R")


def source(name):
    with open(os.path.join(CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def kernels():
    """(file, parameter list, body) of every kernel that begins with grid_begin()."""
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        text = source(name)
        for m in re.finditer(r"__global__ void(?: __launch_bounds__\([^)]*\))?\s+(\w+)\(([^{;]*)\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            body = text[m.end():i]
            if "grid_begin()" in body:
                yield name, m.group(1), m.group(2), body


def test_every_overlapping_kernel_is_seen():
    names = {k for _, k, _, _ in kernels()}
    assert {"scan_kernel", "norm_kernel", "zero_kernel", "split_II_kcontig", "split_II_kstrided", "split_tri_kcontig",
            "split_tri_kstrided", "combine_I_kernel", "crt_II_kernel"} <= names


def test_no_read_only_pointer_to_produced_data():
    for name, kernel, params, _ in kernels():
        for p in params.split(","):
            var = p.split()[-1].lstrip("*") if p.split() else ""
            assert not (var in PRODUCED and "const" in p and "__restrict__" in p), (name, kernel, p)


@pytest.mark.parametrize("name,functions", [
    ("tri_kernels.cuh", ("combine_patch", "digit_sum_term")), ("gemm_II_tc.cu", ("load_pairs", "crt_II_kernel")),
    ("split_core.cuh", ("exp_from_maxbits",)), ("split.cu", ("exp_from_norm",))])
def test_no_read_only_load_of_produced_data(name, functions):
    text = source(name)
    for f in functions:
        m = re.search(r"\b%s\([^;{]*\)\s*\{" % f, text)
        assert m, (name, f)
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        assert "__ldg(" not in text[m.end():i], (name, f)
