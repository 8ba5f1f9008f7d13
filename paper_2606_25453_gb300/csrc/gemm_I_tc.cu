// gemm_I_tc.cu -- Scheme I on the bf16 tensor cores: the digit triangle of
// tri_core.cuh as tcgen05.mma kind::f16 products with accumulators in tensor
// memory, and the kernel that combines its planes into C.
//
// On sm_103a the 8-bit integer MMA exists only as the warp-level mma.sync
// (about 155 TOP/s).  Recentred digits and digit sums are exact bf16 values,
// their products are exact, and FP32 accumulators hold every partial sum
// exactly over 960 (digits) or 256 (digit sums) K elements, so the triangle
// runs at the bf16 rate and every integer, hence C, is the one the mma.sync
// kernel forms.
//
// Work: items (unit, K chunk, tile) in unit order, so that all CTAs read the
// same pair of planes at a time and the operand tiles are reused from L2 as
// in one plain GEMM (keeping a tile and walking all its plane pairs would
// hold every plane live at once).  Each item leaves its exact int32 sums in
// HBM; the p(p+1)/2 products never leave the chip one by one.  The combine
// kernel reads them once.
//
// The main loop: bf16_gemm.cuh, in its single-CTA form (on pairs the short
// segments of the digit sums wait for their drains: n = 8192, p = 8 took 20.6
// ms instead of 16.8).
#include "bf16_gemm.cuh"
#include "crt_core.cuh"
#include "tri_core.cuh"

namespace emu {
namespace {

using bf16g::kBM;
using bf16g::kBN;
constexpr int64_t kSms = 152;  // SMs of a GB300: layouts do not depend on the handle

struct KParamsTri {
  CUtensorMap tA;  // planes as bytes: 128-byte x 128-row boxes, 128-byte swizzle
  CUtensorMap tB;  // 128-byte x 256-row boxes
  TriPlan tp;
  int nst, kcs, nkc;  // 64-deep chunks of a plane; chunks per K range; K ranges
  int tiles_m, tiles_n;  // 128-row and 256-column tiles
  int M, N;  // rows of A's planes and of B's
  int32_t* Cs;  // output planes, tile by tile (tri_elem)
  int* status;
};

// Output planes are stored tile by tile: element (r, c) of a tile at
// ((c / 4) * 128 + r) * 4 + c % 4, so that a warp of the drain (32 rows, four
// columns) and of the combine kernel both touch whole 128-byte lines.
__host__ __device__ __forceinline__ int64_t tri_elem(int r, int c4) { return (static_cast<int64_t>(c4) * kBM + r) * 4; }
constexpr int64_t kTileElems = static_cast<int64_t>(kBM) * kBN;

// Work items (unit, K range, tile) in that order; a unit's plane pairs.
struct TriWork {
  const KParamsTri& kp;
  __device__ __forceinline__ int nitems() const {
    return kp.tp.nunits * kp.nkc * kp.tiles_m * kp.tiles_n;
  }
  __device__ __forceinline__ bf16g::Item item(int i) const {
    const int tiles = kp.tiles_m * kp.tiles_n, per = kp.nkc * tiles;
    bf16g::Item t;
    t.unit = i / per;
    i -= t.unit * per;
    t.aux = i / tiles;  // K range
    tile_coords16(i - t.aux * tiles, kp.tiles_m, kp.tiles_n, t.tm, t.tn);
    const TriUnit u = kp.tp.unit[t.unit];
    t.np = u.count;
    t.seg = u.sums ? bf16g::Cfg<false>::kSeg16 : bf16g::Cfg<false>::kSeg14;
    t.k0 = t.aux * kp.kcs;
    t.k1 = t.k0 + kp.kcs < kp.nst ? t.k0 + kp.kcs : kp.nst;
    return t;
  }
  __device__ __forceinline__ int ya(const bf16g::Item& t, int q) const {
    return kp.tp.pa[kp.tp.unit[t.unit].first + q] * kp.M + t.tm * kBM;
  }
  __device__ __forceinline__ int yb(const bf16g::Item& t, int q) const {
    return kp.tp.pb[kp.tp.unit[t.unit].first + q] * kp.N + t.tn * kBN;
  }
  // the last column tile only as many as N needs (MMA widths in steps of 32)
  __device__ __forceinline__ int cols(const bf16g::Item& t) const {
    const int n = kp.N - t.tn * kBN;
    return n >= kBN ? kBN : (n + 31) & ~31;
  }
};

__global__ void __launch_bounds__(bf16g::kThreads, 1) gemm_I_tc_kernel(const __grid_constant__ KParamsTri kp) {
  extern __shared__ uint8_t smem_raw[];
  const bf16g::Ctx c = bf16g::setup<false>(smem_raw);
  const TriWork w{kp};
  if (c.warp == bf16g::kProducerWarp) {
    if (c.lane == 0) bf16g::produce<false>(c, w, &kp.tA, &kp.tB, kp.status);
    __syncwarp();
  } else if (c.warp == bf16g::kMmaWarp) {
    if (c.lane == 0) bf16g::issue<false>(c, w, kp.status);
    __syncwarp();
  } else {
    // drain: add each finished segment to this thread's exact int32 sums
    constexpr int kC = bf16g::kDrainCols;
    const int c0 = (c.warp >> 2) * kC, row = (c.warp & 3) * 32 + c.lane;
    const uint32_t addr = bf16g::drain_addr(c);
    const int nitems = w.nitems();
    uint32_t seg = 0;
    bool stop = false;
    for (int r = 0; r * c.ncl < nitems && !stop; ++r) {
      const int i = bf16g::item_index(r, c.cid, c.ncl);
      if (i >= nitems) continue;
      const bf16g::Item t = w.item(i);
      const int nseg = (bf16g::stages_of<false>(t) + t.seg - 1) / t.seg;
      const int cols = w.cols(t) - c0;  // of this warp's kC columns
      int run[kC];
#pragma unroll
      for (int x = 0; x < kC; ++x) run[x] = 0;
      for (int s = 0; s < nseg; ++s, ++seg) {
        if (!bf16g::wait_segment(c, seg, kp.status)) {
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
      if (t.tm * kBM + row < kp.M) {
        const int64_t plane = static_cast<int64_t>(kp.tp.unit[t.unit].out) * kp.nkc + t.aux;
        int32_t* dst =
            kp.Cs + (plane * kp.tiles_m * kp.tiles_n + static_cast<int64_t>(t.tn) * kp.tiles_m + t.tm) * kTileElems;
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

// ---------------------------------------------------------------- combine
struct KParamsTriComb {
  const int32_t* Cs;
  int nkc, tiles_m, tiles_n, M, N;
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

// A block combines 32 x 32 outputs, a thread four columns of a row:
// S = sum_s 256^(p-1-s) T_s + R + Q from the planes, rounded once to
// binary64, scaled and updated.  HBM bound: 4 bytes per plane and output
// read (15 planes at p = 8), C written.  All planes are loaded before the
// arithmetic, so that a thread waits for memory once, not once per plane.
template <int P, bool ONE>
__global__ void __launch_bounds__(256) combine_I_kernel(const __grid_constant__ KParamsTriComb kp) {
  using O = TriOut<P, ONE>;
  __shared__ __int128 sR[kCombRows], sQ[kCombCols];
  constexpr int kPC = kBN / kCombCols, kPR = kBM / kCombRows;
  const int tile = blockIdx.x / (kPC * kPR), part = blockIdx.x % (kPC * kPR);
  const int tm = tile % kp.tiles_m, tn = tile / kp.tiles_m;
  const int rt = (part / kPC) * kCombRows, ct = (part % kPC) * kCombCols;  // the patch within the tile
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
      v[u] = live ? __ldg(reinterpret_cast<const int4*>(src + static_cast<int64_t>(u) * kp.nkc * plane))
                  : make_int4(0, 0, 0, 0);
    if (kc == 0) {  // the row and column terms while the planes are on their way
      if (threadIdx.x < kCombRows) {
        const int rr = row0 + threadIdx.x;
        sR[threadIdx.x] = rr < kp.M ? digit_sum_term<P>(kp.sumA + rr, kp.M) : 0;
      } else if (threadIdx.x < kCombRows + kCombCols) {
        const int c = col0 + threadIdx.x - kCombRows;
        const __int128 k0 = static_cast<__int128>((static_cast<unsigned __int128>(kp.const_hi) << 64) | kp.const_lo);
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
  const int erow = kp.EA[row] + kp.escale;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (col + q >= kp.N) break;
    const __int128 t = S[q] + sR[r] + sQ[cl + q];
    const double x = scale2_fast(i128_to_double_rn(t), erow + kp.FB[col + q]);
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

// ---------------------------------------------------------------- plan
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
const TriPlan& plan_of(int p, bool one) { return kPlans.t[one ? 1 : 0][p]; }

template <int P>
cudaError_t launch_combine(const KParamsTriComb& kp, bool one, cudaStream_t st) {
  const unsigned grid =
      static_cast<unsigned>(kp.tiles_m * kp.tiles_n * (kBN / kCombCols) * (kBM / kCombRows));
  if (one)
    combine_I_kernel<P, true><<<grid, 256, 0, st>>>(kp);
  else
    combine_I_kernel<P, false><<<grid, 256, 0, st>>>(kp);
  return cudaGetLastError();
}

template <int P>
void preload_p() {
  cudaFuncAttributes a;
  cudaFuncGetAttributes(&a, combine_I_kernel<P, false>);
  cudaFuncGetAttributes(&a, combine_I_kernel<P, true>);
  if constexpr (P < kTriMaxP) preload_p<P + 1>();
}

}  // namespace

void preload_tri() {
  cudaFuncAttributes a;
  cudaFuncGetAttributes(&a, gemm_I_tc_kernel);
  preload_p<1>();
  preload_split_tri();
  cudaGetLastError();
}

int tri_tile_m() { return kBM; }
int tri_tile_n() { return kBN; }
int tri_num_planes(int p) {
  constexpr PlaneCounts counts{};
  return counts.n[p];
}

TriLayout tri_layout(int64_t M, int64_t N, int64_t k, int p) {
  TriLayout L{};
  L.tiles_m = (M + kBM - 1) / kBM;
  L.tiles_n = (N + kBN - 1) / kBN;
  L.kpad = (k + 63) / 64 * 64;
  const int64_t nst = L.kpad / 64;
  // One unit per s and kind (fewest planes) when its items fill the GPU
  // several times; one unit per plane pair for smaller products, whose time
  // is the longest item's.
  L.one = L.tiles_m * L.tiles_n * plan_of(p, false).nunits < 4 * kSms;
  const TriPlan& tp = plan_of(p, L.one);
  const int most = tp.unit[0].count;
  // int32 sums: most * K * 2^16 < 2^31 bounds the K chunk
  const int64_t lim = ((int64_t{1} << 31) - 1) / (static_cast<int64_t>(most) << 16) / 64;
  L.nkc = (nst + lim - 1) / lim;
  L.kcs = L.nkc > 0 ? (nst + L.nkc - 1) / L.nkc : 0;
  L.planes = static_cast<int64_t>(tp.nunits) * L.nkc;
  L.Cs_bytes = static_cast<size_t>(L.planes) * static_cast<size_t>(L.tiles_m * L.tiles_n) * kTileElems * sizeof(int32_t);
  return L;
}

cudaError_t launch_gemm_I_tc(int p, int out_mode, const GemmTriArgs& a, cudaStream_t st, int part) {
  const TriPlan& tp = plan_of(p, a.L.one);
  const int tiles_m = static_cast<int>(a.L.tiles_m), tiles_n = static_cast<int>(a.L.tiles_n);
  const int nkc = static_cast<int>(a.L.nkc);
  if (tiles_m == 0 || tiles_n == 0 || nkc == 0) return cudaSuccess;
  if (part & 1) {
    KParamsTri kp;
    kp.tA = *a.descA;
    kp.tB = *a.descB;
    kp.tp = tp;
    kp.nst = static_cast<int>(a.L.kpad / 64);
    kp.kcs = static_cast<int>(a.L.kcs);
    kp.nkc = nkc;
    kp.tiles_m = tiles_m;
    kp.tiles_n = tiles_n;
    kp.M = a.M;
    kp.N = a.N;
    kp.Cs = a.Cs;
    kp.status = a.status;
    const int64_t nitems = static_cast<int64_t>(tp.nunits) * nkc * tiles_m * tiles_n;
    const cudaError_t e = bf16g::launch<false>(gemm_I_tc_kernel, nitems, a.num_sms, st, kp);
    if (e != cudaSuccess) return e;
  }
  if (!(part & 2)) return cudaSuccess;
  KParamsTriComb kc;
  kc.Cs = a.Cs;
  kc.nkc = nkc;
  kc.tiles_m = tiles_m;
  kc.tiles_n = tiles_n;
  kc.M = a.M;
  kc.N = a.N;
  kc.sumA = a.sumA;
  kc.sumB = a.sumB;
  // 2^14 K sum_{i,j>=1, i+j<p} 256^(p-1-i-j): s - 1 pairs with i + j = s
  unsigned __int128 w = 0;
  for (int s = 0; s < p; ++s) w = w * 256 + static_cast<unsigned>(s > 1 ? s - 1 : 0);
  w = w * static_cast<unsigned __int128>(a.K) << 14;
  kc.const_lo = static_cast<uint64_t>(w);
  kc.const_hi = static_cast<uint64_t>(w >> 64);
  kc.EA = a.EA;
  kc.FB = a.FB;
  kc.escale = -14 - 8 * (p - 1);
  kc.alpha = a.alpha;
  kc.beta = a.beta;
  kc.C = a.C;
  kc.ldc = a.ldc;
  kc.f32 = out_mode == OUT_F32;
  kc.plain = a.alpha == 1.0 && a.beta == 0.0;
#define EMU_TRI(PP) \
  case PP:          \
    return launch_combine<PP>(kc, a.L.one, st);
  switch (p) {
    EMU_TRI(1) EMU_TRI(2) EMU_TRI(3) EMU_TRI(4) EMU_TRI(5) EMU_TRI(6)
    EMU_TRI(7) EMU_TRI(8) EMU_TRI(9) EMU_TRI(10) EMU_TRI(11) EMU_TRI(12)
    default:
      return cudaErrorInvalidValue;
  }
#undef EMU_TRI
}

}  // namespace emu
