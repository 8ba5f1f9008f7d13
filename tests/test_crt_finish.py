"""The CRT finish of csrc/crt_core.cuh, compiled for the host from the same
source, against exact integers for every number of moduli: x of the symmetric
range (-P/2, P/2] rounded once to binary64, with x next to 0 and next to a
half of P, where the quotient comes from the exact comparison (a product
reaches that branch only for one to three moduli)."""
import ctypes
import os
import random
import shutil
import subprocess

import pytest

import paper_2606_25453_gb300 as emu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2606_25453_gb300", "csrc")
LIB = os.path.join(ROOT, "paper_2606_25453_gb300", "_build", "libemugemm.so")
MAXP, LIMBS = 10, 5

HARNESS = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda.h>
#include <cuda_runtime.h>
// the device functions that the header names, for the host compiler
static inline unsigned __cvta_generic_to_shared(const void*) { return 0; }
static inline int atomicOr(int* p, int v) { int o = *p; *p |= v; return o; }
static inline long long clock64() { return 0; }
static inline long long __double_as_longlong(double x) { long long r; std::memcpy(&r, &x, 8); return r; }
static inline double __longlong_as_double(long long x) { double r; std::memcpy(&r, &x, 8); return r; }
static inline float __uint_as_float(unsigned x) { float r; std::memcpy(&r, &x, 4); return r; }
static inline int __clzll(long long x) { return x ? __builtin_clzll(x) : 64; }
static inline uint64_t __umul64hi(uint64_t a, uint64_t b) {
  return static_cast<uint64_t>((static_cast<unsigned __int128>(a) * b) >> 64);
}
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
#include "crt_core.cuh"
template <int L>
static double run(const uint32_t* x, const emu::CrtPairTables& t) {
  emu::CrtPair<L> a;
  for (int j = 0; j < L; ++j) a.s[j] = 0;
  for (int i = 0; 2 * i < t.nm; ++i)
    for (int j = 0; j < L; ++j) a.s[j] += static_cast<uint64_t>(t.w[i][j]) * x[i];
  return emu::crt_finish_pair<L>(a, t);
}
extern "C" double finish(const uint32_t* x, const emu::CrtPairTables* t) {
  switch (t->limbs) {
    case 2: return run<2>(x, *t);
    case 3: return run<3>(x, *t);
    case 4: return run<4>(x, *t);
    default: return run<5>(x, *t);
  }
}
extern "C" int table_bytes() { return static_cast<int>(sizeof(emu::CrtPairTables)); }
"""


class Tables(ctypes.Structure):
    _fields_ = [("c", ctypes.c_uint32 * MAXP), ("off", ctypes.c_uint32 * MAXP),
                ("w", (ctypes.c_uint32 * LIMBS) * MAXP), ("P", ctypes.c_uint32 * LIMBS),
                ("Phalf", ctypes.c_uint32 * LIMBS), ("recip", ctypes.c_uint64), ("sh", ctypes.c_int32),
                ("frac", ctypes.c_int32), ("limbs", ctypes.c_int32), ("nm", ctypes.c_int32)]


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    cxx = shutil.which("g++")
    inc = next((d for d in ("/usr/local/cuda/include", "/usr/include") if
                os.path.exists(os.path.join(d, "cuda_runtime.h"))), None)
    if not cxx or not inc:
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("crt")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-fPIC", "-shared", "-I", inc, "-I", CSRC,
                    str(d / "h.cpp"), "-o", str(d / "h.so")], check=True)
    h = ctypes.CDLL(str(d / "h.so"))
    h.finish.restype = ctypes.c_double
    assert h.table_bytes() == ctypes.sizeof(Tables)
    tables = ctypes.CDLL(LIB)._ZN3emu20host_crt_pair_tablesEiPNS_13CrtPairTablesE
    return h, tables


@pytest.mark.parametrize("nm", range(1, 21))
def test_finish_is_exact(host, nm):
    h, build = host
    t = Tables()
    build(nm, ctypes.byref(t))
    arr = (ctypes.c_int32 * nm)()
    assert emu.emu_moduli(nm, arr) == nm
    mods = list(arr)
    P = 1
    for m in mods:
        P *= m
    rng = random.Random(nm)
    xs = list(range(-3, 4)) + [rng.randrange(-(P // 2) + 1, P // 2 + 1) for _ in range(200)]
    # beside a half: from the last integer to well past the width of the exact comparison
    for d in list(range(0, 40)) + [P >> s for s in range(3, 60)] + [rng.randrange(1 + (P >> 27)) for _ in range(60)]:
        xs += [P // 2 - d, -(P // 2) + 1 + d]
    # beside powers of two, where binary64 rounds and carries
    for b in range(50, P.bit_length() - 1):
        xs += [s * ((1 << b) + d) for s in (1, -1) for d in (-1, 0, 1)]
    for x in xs:
        if not -(P // 2) < x <= P // 2 and not (P % 2 and x == -(P // 2)):
            continue
        for form in range(2):
            v = (ctypes.c_uint32 * MAXP)()
            for i in range((nm + 1) // 2):
                m = mods[2 * i:2 * i + 2]
                co = (t.c[i] & 0xFFFF, t.c[i] >> 16)
                r = [x % q for q in m]
                if form:  # the 3M form: a difference of two residues, kept non-negative
                    r2 = [rng.randrange(q) for q in m]
                    r1 = [(a + b) % q for a, b, q in zip(r, r2, m)]
                    v[i] = sum(a * c for a, c in zip(r1, co)) + t.off[i] - sum(a * c for a, c in zip(r2, co))
                else:
                    v[i] = sum(a * c for a, c in zip(r, co))
            assert h.finish(v, ctypes.byref(t)) == float(x), (nm, x, form)
