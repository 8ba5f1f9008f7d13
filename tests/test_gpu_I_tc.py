"""Scheme I on the bf16 tensor cores: digit products, digit-sum products and
the combine kernel give the oracle's result bit for bit.  The exact integers
fix every rounding, so the tolerance is zero."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_25453_gb300 as emu  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def run(orc, A, B, p, alpha=1.0, beta=0.0, C0=None):
    h = emu.Handle(0)
    C = dev(C0) if C0 is not None else None
    got = emu.dgemm(dev(A), dev(B), C, alpha, beta, scheme="I", p=p, handle=h).cpu().numpy()
    assert h.status() == 0
    h.close()
    assert np.array_equal(got, orc.emu_I(A, B, p, alpha=alpha, beta=beta, C=C0))


# one element; tile edges (128 rows, 256 columns) and their neighbours; K at
# and around a 64-deep stage, a 256-deep digit-sum segment, a 960-deep digit
# segment and several of both
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (127, 255, 63), (128, 256, 64), (129, 257, 65), (3, 300, 256),
                                   (200, 17, 257), (130, 33, 960), (40, 600, 1025), (5, 7, 4100)])
@pytest.mark.parametrize("p", [1, 2, 3, 8, 12])
def test_tile_and_segment_edges(orc, m, n, k, p):
    A, B = synth.gemm_pair(m, n, k, 1.0, 11 * m + n + k + p)
    run(orc, A, B, p)


@pytest.mark.parametrize("p", range(1, 13))
def test_every_slice_count_with_update(orc, p):
    A, B = synth.gemm_pair(150, 270, 700, 2.0, 40 + p)
    run(orc, A, B, p, alpha=-1.5, beta=0.25, C0=synth.test_matrix(150, 270, 1.0, 90 + p))


# more than eight slices take this path from 2^33 multiply-adds on: a few rows
# against many columns at that size
@pytest.mark.parametrize("p", [9, 12])
def test_many_slices_large_product(orc, p):
    m, n, k = 66, 16400, 7990
    A, B = synth.gemm_pair(m, n, k, 2.0, 60 + p)
    h = emu.Handle(0)
    got = emu.dgemm(dev(A), dev(B), scheme="I", p=p, handle=h).cpu().numpy()
    assert h.status() == 0
    h.close()
    rows = [0, 37, 65]
    assert np.array_equal(got[rows], orc.emu_I(A[rows], B, p))


# every digit at an end of its range: all-ones bytes (tails 255 -> +127),
# zero tails (-128), and the most negative leading digit, over K chunks of
# the int32 sums (12 slices: five pairs share one sum below K = 6528)
@pytest.mark.parametrize("a", [1.0 - 2.0 ** -53, 0.5, -0.5, -(1.0 - 2.0 ** -53)])
def test_extreme_digits(orc, a):
    A = np.full((3, 9000), a)
    B = np.full((9000, 5), -a)
    for p in (7, 8, 12):
        run(orc, A, B, p)


# digit sums at -256 over whole 256-deep segments with one -255 in each, on
# both sides: every segment's FP32 sum ends at 2^24 - 511, an odd integer
# beside the end of the exact range (constant operands give even sums only)
@pytest.mark.parametrize("p", [3, 4, 6])
def test_odd_sums_beside_2_24(orc, p):
    k = 1024
    rng = np.random.Generator(np.random.PCG64(p))
    low = -(2.0 ** (8 * p - 1)) + 1  # leading digit -128, bytes 0 .. 0 1: digits -128, .., -128, -127
    A, B = np.full((140, k), low), np.full((k, 270), low)
    for seg in range(0, k, 256):
        at = seg + int(rng.integers(256))
        A[:, at] += 2.0 ** (8 * (p - 2))  # second byte 1: digit sum -255
        B[at, :] += 2.0 ** (8 * (p - 2))
    assert 255 * 65536 + 255 * 255 == 2 ** 24 - 511
    run(orc, A, B, p)


def test_one_plane_per_group_and_row_strides(orc):
    # enough tiles that each group of digit sums shares one output plane
    A, B = synth.gemm_pair(1300, 2200, 130, 0.5, 77)
    h = emu.Handle(0)
    Ap = torch.full((1300, 133), float("nan"), dtype=torch.float64, device="cuda")
    Ap[:, :130] = dev(A)
    Bp = torch.full((130, 2201), float("nan"), dtype=torch.float64, device="cuda")
    Bp[:, :2200] = dev(B)
    C = emu.dgemm(Ap[:, :130], Bp[:, :2200], scheme="I", p=8, handle=h).cpu().numpy()
    assert h.status() == 0
    h.close()
    assert np.array_equal(C, orc.emu_I(A, B, 8))


def test_small_workspace_keeps_the_int8_kernel(orc):
    # a caller's workspace that holds the slices but not the digit planes
    m, n, k, p = 140, 90, 300, 7
    A, B = synth.gemm_pair(m, n, k, 1.0, 5)
    h = emu.Handle(0)
    full = ctypes.c_size_t()
    emu.check(emu.emu_workspace_size(1, m, n, k, p, 0, ctypes.byref(full)))
    rows = emu.emu_split_rows(m) + emu.emu_split_rows(n)
    small = rows * emu.emu_split_cols_I(k, p) + 4 * 4096
    assert small < full.value
    want = orc.emu_I(A, B, p)
    for size in (small, full.value):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        emu.check(emu.emu_set_workspace(h.h, ws.data_ptr(), size))
        got = emu.dgemm(dev(A), dev(B), scheme="I", p=p, handle=h).cpu().numpy()
        assert h.status() == 0 and np.array_equal(got, want)
    h.close()


CHILD = r"""
import sys
sys.path.insert(0, %r)
import numpy as np, torch
import paper_2606_25453_gb300 as emu, synth
h = emu.Handle(0)
A, B = synth.gemm_pair(300, 260, 1100, 1.0, 8)
C = emu.dgemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), scheme="I", p=8, handle=h)
assert h.status() == 0
np.save(sys.argv[1], C.cpu().numpy())
"""


def test_engine_switch_gives_the_same_bits(orc, tmp_path):
    A, B = synth.gemm_pair(300, 260, 1100, 1.0, 8)
    out = str(tmp_path / "c.npy")
    r = subprocess.run([sys.executable, "-c", CHILD % ROOT, out], env=dict(os.environ, EMU_I_ENGINE="mma"),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert np.array_equal(np.load(out), orc.emu_I(A, B, 8))
    run(orc, A, B, 8)


# products narrower than a tile: boxes and combine blocks follow M in steps of
# 8 and 32 rows, N in steps of 32 columns
@pytest.mark.parametrize("m,n", [(1, 300), (300, 1), (8, 32), (9, 33), (121, 31), (136, 64), (33, 250), (127, 255)])
def test_narrow_products(orc, m, n):
    A, B = synth.gemm_pair(m, n, 200, 1.0, 10 * m + n)
    C0 = synth.test_matrix(m, n, 1.0, m + n)
    for p in (2, 8):
        run(orc, A, B, p, alpha=-0.5, beta=2.0, C0=C0)


# both sides of every line between the bf16 engine and the INT8 kernel for
# long, narrow products of short K (and short, wide ones): rows for 20 items
# per SM, columns times K, the single columns of three slices
@pytest.mark.parametrize("m,n,k,p,layout,bf16", [
    (26000, 8, 32, 8, "row", False), (25000, 8, 32, 8, "row", True), (26000, 8, 128, 8, "row", False),
    (26000, 8, 129, 8, "row", True), (26000, 64, 32, 8, "row", False), (26000, 65, 32, 8, "row", True),
    (26000, 33, 63, 8, "row", True), (26000, 32, 63, 7, "row", True), (31000, 32, 63, 7, "row", False), (8, 26000, 40, 8, "col", False),
    (7, 52000, 32, 8, "row", False), (9, 52000, 32, 8, "row", True), (7, 52000, 33, 8, "row", True),
    (97300, 8, 64, 3, "row", False), (97300, 9, 64, 3, "row", True), (97300, 3, 64, 2, "row", True)])
def test_engine_lines_of_narrow_products(orc, m, n, k, p, layout, bf16):
    A, B = synth.gemm_pair(m, n, k, 1.0, m + n + k)
    h = emu.Handle(0)
    Ad, Bd = (dev(A), dev(B)) if layout == "row" else (dev(A.T).t(), dev(B.T).t())
    C = torch.empty((m, n), dtype=torch.float64, device="cuda") if layout == "row" else \
        torch.empty((n, m), dtype=torch.float64, device="cuda").t()
    h.trace(True)
    h.trace_read()
    emu.dgemm(Ad, Bd, C, scheme="I", p=p, handle=h)
    t = h.trace_read()
    h.trace(False)
    assert h.status() == 0
    assert (t["ms_other"] > 0.0) == bf16  # the combine kernel is the bf16 engine's
    h.close()
    rows = np.unique(np.linspace(0, m - 1, 700).astype(int))
    cols = np.unique(np.linspace(0, n - 1, 700).astype(int))
    want = orc.emu_I(np.ascontiguousarray(A[rows]), np.ascontiguousarray(B[:, cols]), p)
    assert np.array_equal(C.cpu().numpy()[np.ix_(rows, cols)], want)
