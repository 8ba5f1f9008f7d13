// tri_kernels.cuh -- the digit triangle of tri_core.cuh on the device: its
// unit tables, the layout of its output planes and their combination into C,
// shared by the single and the grouped products.
#pragma once
#include "bf16_gemm.cuh"
#include "crt_core.cuh"
#include "emu_internal.h"
#include "tri_core.cuh"

namespace emu {
namespace {

using bf16g::kBM;
using bf16g::kBN;
constexpr int64_t kSms = 152;  // SMs of a GB300: layouts do not depend on the handle

// Output planes are stored tile by tile: element (r, c) of a tile at
// ((c / 4) * 128 + r) * 4 + c % 4, so that a warp of the drain (32 rows, four
// columns) and of the combine kernel both touch whole 128-byte lines.
__host__ __device__ __forceinline__ int64_t tri_elem(int r, int c4) { return (static_cast<int64_t>(c4) * kBM + r) * 4; }
constexpr int64_t kTileElems = static_cast<int64_t>(kBM) * kBN;

// The units of the triangle, longest first: one per group (one false) or one
// per plane pair (one true).
constexpr TriPlan make_plan(int p, bool one) {
  TriPlan tp{};
  int np = 0, out = 0;
  for (int s = 0; s <= p + 1; ++s) {  // s < p: digit sums of s; p: the diagonal; p + 1: the direct pair
    int first = np;
    const int npairs = s < p ? (s + 1) / 2 : s == p ? tri_diag(p) : (p > 1 ? 2 : 0);
    for (int i = 0; i < npairs; ++i) {
      if (s < p) {
        if (i == 0 && s == p - 1) continue;
        tp.pa[np] = tp.pb[np] = static_cast<uint8_t>(tri_cross_plane(p, i, s - i));
      } else if (s == p) {
        tp.pa[np] = tp.pb[np] = static_cast<uint8_t>(i);
      } else {
        tp.pa[np] = static_cast<uint8_t>(i == 0 ? 0 : p - 1);
        tp.pb[np] = static_cast<uint8_t>(i == 0 ? p - 1 : 0);
      }
      ++np;
      if (one || s == p || i + 1 == npairs) {
        TriUnit& u = tp.unit[tp.nunits++];
        u.first = static_cast<uint8_t>(first);
        u.count = static_cast<uint8_t>(np - first);
        u.sums = s < p;
        u.out = static_cast<uint8_t>(out++);
        first = np;
      }
    }
  }
  // longest first (stable): the short units fill the last wave
  for (int a = 1; a < tp.nunits; ++a)
    for (int b = a; b > 0 && tp.unit[b].count > tp.unit[b - 1].count; --b) {
      const TriUnit t = tp.unit[b];
      tp.unit[b] = tp.unit[b - 1];
      tp.unit[b - 1] = t;
    }
  return tp;
}

// Built by the compiler: planning a call is part of its launch latency.
struct PlanTable {
  TriPlan t[2][kTriMaxP + 1];
};
constexpr PlanTable make_table() {
  PlanTable x{};
  for (int p = 1; p <= kTriMaxP; ++p) {
    x.t[0][p] = make_plan(p, false);
    x.t[1][p] = make_plan(p, true);
  }
  return x;
}
constexpr PlanTable kPlans = make_table();
struct PlaneCounts {
  int n[kTriMaxP + 1] = {};
  constexpr PlaneCounts() {
    for (int p = 1; p <= kTriMaxP; ++p) n[p] = tri_planes(p);
  }
};
inline const TriPlan& plan_of(int p, bool one) { return kPlans.t[one ? 1 : 0][p]; }

// The products of a work list: every item's exact int32 sums to the tile that
// w.tile_of names.
template <class W>
__device__ __forceinline__ void tri_gemm(const W& w, int* status) {
  extern __shared__ uint8_t smem_raw[];
  const bf16g::Ctx c = bf16g::setup<false>(smem_raw);
  if (c.warp == bf16g::kProducerWarp) {
    if (c.lane == 0) bf16g::produce<false>(c, w, status);
    __syncwarp();
  } else if (c.warp == bf16g::kMmaWarp) {
    if (c.lane == 0) bf16g::issue<false>(c, w, status);
    __syncwarp();
  } else {
    // drain: add each finished segment to this thread's exact int32 sums
    constexpr int kC = bf16g::kDrainCols;
    const int c0 = (c.warp >> 2) * kC, row = (c.warp & 3) * 32 + c.lane;
    const uint32_t addr = bf16g::drain_addr(c);
    uint32_t seg = 0;
    bool stop = false;
    bf16g::Item t;
    for (int r = 0; !stop && w.at(r, c.cid, c.ncl, t); ++r) {
      const int nseg = (bf16g::stages_of<false>(t) + t.seg - 1) / t.seg;
      const int cols = t.cols - c0;  // of this warp's kC columns
      int run[kC];
#pragma unroll
      for (int x = 0; x < kC; ++x) run[x] = 0;
      for (int s = 0; s < nseg; ++s, ++seg) {
        if (!bf16g::wait_segment(c, seg, status)) {
          stop = true;
          break;
        }
#pragma unroll
        for (int q = 0; q < kC / 16; ++q) {
          uint32_t v[16];
          if (16 * q < cols) {
            tmem_ld16(addr + (seg & 1u) * kBN + 16 * q, v);
            tmem_wait_ld();
          }
          if (q == kC / 16 - 1) bf16g::release_segment<false>(c, seg);
          if (16 * q < cols) {
#pragma unroll
            for (int x = 0; x < 16; ++x) run[16 * q + x] += __float2int_rn(__uint_as_float(v[x]));
          }
        }
      }
      if (stop) break;
      if (t.tm * kBM + row < w.rows(t)) {
        int32_t* const dst = w.tile_of(t);
#pragma unroll
        for (int g = 0; g < kC / 4; ++g)
          if (4 * g < cols)
            *reinterpret_cast<int4*>(dst + tri_elem(row, c0 / 4 + g)) =
                make_int4(run[4 * g], run[4 * g + 1], run[4 * g + 2], run[4 * g + 3]);
      }
    }
  }
  bf16g::finish<false>(c);
}

struct KParamsTriComb {
  const int32_t* Cs;
  int nkc, tiles_m, tiles_n, M, N;
  int pr, pc;  // patches per tile (patch_rows, patch_cols)
  const int32_t* sumA;  // digit sums of A's rows: digit t of row r at [t * M + r]
  const int32_t* sumB;
  uint64_t const_lo, const_hi;  // the products of the 128s alone (128-bit)
  const int32_t* EA;
  const int32_t* FB;
  int escale;
  double alpha, beta;
  void* C;
  int64_t ldc;
  int plain;  // alpha = 1, beta = 0
  int f32;    // C is binary32
};

// 128 sum_t U_t (256^(p-1-t) - 1) / 255 from the digit sums U_t of one row or
// column: with V_t = U_0 + .. + U_t it is 128 sum_{t<p-1} V_t 256^(p-2-t).
template <int P>
__device__ __forceinline__ __int128 digit_sum_term(const int32_t* U, int64_t stride) {
  __int128 r = 0;
  long long v = 0;
#pragma unroll
  for (int t = 0; t + 1 < P; ++t) {
    v += U[t * stride];
    r = r * 256 + v;
  }
  return r * 128;
}

// Plane of c(0, 0) and of the direct pair among the output planes of one K
// chunk, and the planes per digit-sum group: with one unit per group (ONE
// false) or one per plane pair (ONE true), as make_plan lays them out.
template <int P, bool ONE>
struct TriOut {
  static constexpr int pairs(int s) {  // digit-sum pairs (i, j) with i + j = s
    int n = 0;
    for (int i = 0; 2 * i < s; ++i) n += !(i == 0 && s == P - 1);
    return n;
  }
  static constexpr int nx(int s) { return ONE ? pairs(s) : (pairs(s) > 0 ? 1 : 0); }
  static constexpr int xoff(int s) {
    int n = 0;
    for (int q = 0; q < s; ++q) n += nx(q);
    return n;
  }
  static constexpr int doff = xoff(P), diroff = doff + tri_diag(P);
  static constexpr int ndir = P > 1 ? (ONE ? 2 : 1) : 0;
  static constexpr int planes = diroff + ndir;
};

constexpr int kCombRows = 32, kCombCols = 32;  // a combine block's patch: one 8 x 16 piece per warp
// Patches of one tile that a block is launched for: of a product narrower
// than a tile only those it has (3000 products of 32 x 32: 31 of 32 blocks
// had nothing to do, 0.37 ms of 1.13).
__host__ __device__ __forceinline__ int patch_rows(int64_t m) {
  return static_cast<int>(((m < kBM ? m : kBM) + kCombRows - 1) / kCombRows);
}
__host__ __device__ __forceinline__ int patch_cols(int64_t n) {
  return static_cast<int>(((n < kBN ? n : kBN) + kCombCols - 1) / kCombCols);
}

// A block combines 32 x 32 outputs, a thread four columns of a row:
// S = sum_s 256^(p-1-s) T_s + R + Q from the planes, rounded once to
// binary64, scaled and updated.  HBM bound: 4 bytes per plane and output
// read (15 planes at p = 8), C written.  All planes are loaded before the
// arithmetic, so that a thread waits for memory once, not once per plane.
template <int P, bool ONE>
__device__ __forceinline__ void combine_patch(const KParamsTriComb& kp, int block) {
  using O = TriOut<P, ONE>;
  __shared__ __int128 sR[kCombRows], sQ[kCombCols];
  __shared__ int sE[kCombRows], sF[kCombCols];
  constexpr int kPC = kBN / kCombCols, kPR = kBM / kCombRows;
  int tile, pr, pc;  // the patch within the tile
  if (kp.pr * kp.pc == kPR * kPC) {  // whole tiles: constant divisors
    tile = block / (kPC * kPR);
    const int part = block % (kPC * kPR);
    pr = part / kPC;
    pc = part % kPC;
  } else {
    tile = block / (kp.pr * kp.pc);
    const int part = block - tile * kp.pr * kp.pc;
    pr = part / kp.pc;
    pc = part - pr * kp.pc;
  }
  const int tm = tile % kp.tiles_m, tn = tile / kp.tiles_m;
  const int rt = pr * kCombRows, ct = pc * kCombCols;
  const int row0 = tm * kBM + rt, col0 = tn * kBN + ct;
  if (row0 >= kp.M || col0 >= kp.N) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = (warp >> 1) * 8 + (lane >> 2), cl = (warp & 1) * 16 + (lane & 3) * 4;
  const int row = row0 + r, col = col0 + cl;
  const bool live = row < kp.M && col < kp.N;
  const int64_t plane = static_cast<int64_t>(kp.tiles_m) * kp.tiles_n * kTileElems;
  const int32_t* src = kp.Cs + static_cast<int64_t>(tile) * kTileElems + tri_elem(rt + r, (ct + cl) / 4);
  __int128 S[4] = {0, 0, 0, 0};
  for (int kc = 0; kc < kp.nkc; ++kc, src += plane) {
    int4 v[O::planes];
#pragma unroll
    for (int u = 0; u < O::planes; ++u)
      v[u] = live ? __ldcg(reinterpret_cast<const int4*>(src + static_cast<int64_t>(u) * kp.nkc * plane))
                  : make_int4(0, 0, 0, 0);
    if (kc == 0) {  // the row and column terms while the planes are on their way
      if (threadIdx.x < kCombRows) {
        const int rr = row0 + threadIdx.x;
        sE[threadIdx.x] = rr < kp.M ? kp.EA[rr] + kp.escale : 0;
        sR[threadIdx.x] = rr < kp.M ? digit_sum_term<P>(kp.sumA + rr, kp.M) : 0;
      } else if (threadIdx.x < kCombRows + kCombCols) {
        const int c = col0 + threadIdx.x - kCombRows;
        const __int128 k0 = static_cast<__int128>((static_cast<unsigned __int128>(kp.const_hi) << 64) | kp.const_lo);
        sF[threadIdx.x - kCombRows] = c < kp.N ? kp.FB[c] : 0;
        sQ[threadIdx.x - kCombRows] = (c < kp.N ? digit_sum_term<P>(kp.sumB + c, kp.N) : 0) + k0;
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      auto at = [&](int u) -> long long { return q == 0 ? v[u].x : q == 1 ? v[u].y : q == 2 ? v[u].z : v[u].w; };
      // T_s = x_s - sum over the digit-sum pairs (i, j) of (c(i,i) + c(j,j))
      //       (+ c(s/2, s/2) for even s); the pairs of s cover every i <= s
      //       but s / 2 (and, at s = p - 1, but 0 and p - 1).
      // Four T_s at a time fit one 64-bit sum (|T_s| < 2^33).
      long long pre = 0, part64 = 0;
      __int128 Sq = 0;
#pragma unroll
      for (int s = 0; s < P; ++s) {
        long long T = 0;
#pragma unroll
        for (int x = 0; x < O::nx(s); ++x) T += at(O::xoff(s) + x);
        if (s < tri_diag(P)) pre += at(O::doff + s);
        if (s + 1 == P && P > 1) {
#pragma unroll
          for (int x = 0; x < O::ndir; ++x) T += at(O::diroff + x);
          if (P > 2) T += at(O::doff);
        }
        if (P > 2 || s == 0) {
          if (s % 2 == 0 && s / 2 < tri_diag(P)) T += 2 * at(O::doff + s / 2);
          T -= pre;
        }
        part64 = part64 * 256 + T;
        if (s % 4 == 3 || s + 1 == P) {
          Sq = Sq * (static_cast<__int128>(1) << (8 * (s % 4 + 1))) + part64;
          part64 = 0;
        }
      }
      S[q] += Sq;
    }
  }
  __syncthreads();
  if (!live) return;
  const int erow = sE[r];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (col + q >= kp.N) break;
    const __int128 t = S[q] + sR[r] + sQ[cl + q];
    const double x = scale2_fast(i128_to_double_rn(t), erow + sF[cl + q]);
    if (!kp.f32) {
      double* cp = static_cast<double*>(kp.C) + static_cast<int64_t>(row) * kp.ldc + col + q;
      *cp = kp.plain ? x : blas_update(kp.alpha, x, kp.beta, kp.beta != 0.0 ? *cp : 0.0);
    } else {
      float* cp = static_cast<float*>(kp.C) + static_cast<int64_t>(row) * kp.ldc + col + q;
      *cp = static_cast<float>(
          kp.plain ? x : blas_update(kp.alpha, x, kp.beta, kp.beta != 0.0 ? static_cast<double>(*cp) : 0.0));
    }
  }
}

}  // namespace
}  // namespace emu
