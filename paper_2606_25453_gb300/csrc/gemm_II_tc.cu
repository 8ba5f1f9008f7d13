// gemm_II_tc.cu -- Scheme II on the bf16 tensor cores (tcgen05.mma
// kind::f16) with accumulators in tensor memory, and the CRT.
//
// On sm_103a the 8-bit integer MMA exists only as the warp-level mma.sync.
// The symmetric residues of Eq. (5) (|r| <= 128) are exact bf16 values, the
// products of two of them (|r_a r_b| <= 2^14) are exact, and an FP32 sum of
// up to 960 such products stays an exact integer (|sum| <= 960 * 2^14 <
// 2^24).  So every per-modulus product of Eq. (6) runs as a bf16 GEMM on the
// 5th-generation tensor cores in K segments of 896 (CTA pairs) or 960, and the result is
// bit-identical to the INT8 kernel's.
//
// The work is modulus-major, as in the paper's Scheme II kernel (Sec. IV):
// a persistent kernel walks (modulus, tile) items in that order, so that all
// CTAs work on the same pair of residue planes at the same time and the
// operand tiles are reused from L2 as in one plain GEMM (walking all moduli
// of one tile before the next keeps 16 x more operand data live and reads
// the planes from DRAM about 20 times).  Each item's product stays in TMEM;
// the epilogue reduces it modulo m_l (Eq. 7) and writes only the residue
// bytes (one per output and modulus).  A second kernel then forms the CRT
// sum of Eq. (8) from the residues, reduces it modulo P, lifts it to the
// symmetric range, rounds it once to binary64, scales it back and applies
// the BLAS update (3M combination of Eq. (16) for complex input).
//
// The main loop and its two forms (CTA pairs, single CTAs): bf16_gemm.cuh.
#include <cstdlib>
#include <type_traits>

#include "bf16_gemm.cuh"
#include "crt_core.cuh"

namespace emu {
namespace {

using bf16g::kBM;
using bf16g::kBN;

// Residue GEMM, 14 moduli, single / pair in us: n = 2048, K = 512: 66 / 80,
// 896: 94 / 87, 1024: 112 / 108, 2048: 177 / 161; n = 4096, K = 512: 228 /
// 285, 896: 338 / 299, 3072: 916 / 813; n = 1024, K = 896: 31 / 31.
constexpr int64_t kPairMinK = 896;

struct KParamsIITC {
  CUtensorMap tA;  // bf16 planes as bytes: 128-byte x 128-row boxes, 128-byte swizzle
  CUtensorMap tB;  // 128-byte x (256 or 128)-row boxes
  int nst;         // 64-wide K chunks per plane
  int tiles_m;     // 128-row tiles of the residue matrices (even with CTA pairs)
  int tiles_n;     // 256-column tiles
  int N;
  int nplanes;     // NSET * nm residue planes (plane p = set * nm + l)
  int nm;
  int rowsA_pad, rowsB_pad;
  uint8_t* R;      // residues: plane p, row r, column c at R[(p * tiles_m * 128 + r) * ldr + c]
  int64_t ldr;     // tiles_n * 256
  int* status;
};

// Segments (|sum| <= 2^24 each) between folds of the int32 sums, the largest
// sum that is folded then, and what a fold leaves of it.
constexpr int kFold = 64;
constexpr int64_t kSumMax = (int64_t{kFold} << 24) + (int64_t{1} << 22);
constexpr int64_t kFoldMax = ((kSumMax >> 16) + 1) * 128 + 0xFFFF;

// A multiple of m_l added to (or removed from) an exact int32 sum |x| <=
// kSumMax, keeping its residue: x = hi 2^16 + lo -> hi (2^16 mod m) + lo,
// |result| <= kFoldMax < 2^21.1 (p16: the symmetric residue of 2^16 mod m,
// |p16| <= 128).
static_assert(kSumMax < INT32_MAX && kFoldMax < (int64_t{1} << 22) && kFoldMax < 2580000,
              "folded sums stay in int32, and within what mod4 takes");
__device__ __forceinline__ int fold16(int x, int p16) { return (x >> 16) * p16 + (x & 0xFFFF); }

// Residues in [0, m) of four sums |x| <= 2^21.3 (2.58e6; fold16's output is smaller), one byte
// each, in FP32 arithmetic without conversions or corrections: with x / m =
// n + j / m, y = x / m + 1 / (2m) - 1/2 lies 1 / (2m) >= 0.0019 inside
// (n - 1/2, n + 1/2), and its computed value errs by less than 2^-10 (inv by
// 2^-25 of |x / m| < 2^13.9, the FMA by half an ulp, 2^-11), so rounding y to
// an integer gives n and r = x - n m is exact.
__device__ __forceinline__ uint32_t mod4(const int* x, float inv, float off, float negm) {
  uint32_t r[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    // 1.5 2^23 + x has x in its low mantissa bits
    const float xf = __uint_as_float(0x4B400000u + static_cast<uint32_t>(x[k])) - 12582912.0f;
    const float q = __fadd_rn(__fadd_rn(__fmaf_rn(xf, inv, off), 12582912.0f), -12582912.0f);
    r[k] = __float_as_uint(__fadd_rn(__fmaf_rn(q, negm, xf), 8388608.0f));
  }
  return __byte_perm(__byte_perm(r[0], r[1], 0x0040u), __byte_perm(r[2], r[3], 0x0040u), 0x5410u);
}

// Work item i: plane p = i / (tiles per plane), then the tile.
template <bool PAIR>
struct WorkII {
  const KParamsIITC& kp;
  __device__ __forceinline__ bool at(int r, int cid, int ncl, bf16g::Item& t) const {
    const int tm_units = PAIR ? kp.tiles_m / 2 : kp.tiles_m, per_plane = tm_units * kp.tiles_n;
    const int i = bf16g::item_index(r, cid, ncl);
    if (i >= kp.nplanes * per_plane) return false;
    t.unit = i / per_plane;
    tile_coords16(i - t.unit * per_plane, tm_units, kp.tiles_n, t.tm, t.tn);
    if (PAIR) t.tm *= 2;
    t.np = 1;
    t.k0 = 0;
    t.k1 = kp.nst;
    t.seg = bf16g::Cfg<PAIR>::kSeg14;
    t.cols = bf16g::tile_cols(kp.N, t.tn);
    return true;
  }
  __device__ __forceinline__ int ya(const bf16g::Item& t, int) const { return t.unit * kp.rowsA_pad + t.tm * kBM; }
  __device__ __forceinline__ int yb(const bf16g::Item& t, int) const { return t.unit * kp.rowsB_pad + t.tn * kBN; }
  __device__ __forceinline__ const CUtensorMap* tA(const bf16g::Item&) const { return &kp.tA; }
  __device__ __forceinline__ const CUtensorMap* tB(const bf16g::Item&) const { return &kp.tB; }
  __device__ __forceinline__ int bytes(const bf16g::Item&) const { return bf16g::Cfg<PAIR>::kChunkBytes; }
};

template <bool PAIR>
__global__ void __launch_bounds__(bf16g::kThreads, 1)
    gemm_II_tc_kernel(const __grid_constant__ KParamsIITC kp, const __grid_constant__ ModTables mt) {
  extern __shared__ uint8_t smem_raw[];
  const bf16g::Ctx c = bf16g::setup<PAIR>(smem_raw);
  const WorkII<PAIR> w{kp};
  if (c.warp == bf16g::kProducerWarp) {
    if (c.lane == 0) bf16g::produce<PAIR>(c, w, kp.status);
    __syncwarp();
  } else if (c.warp == bf16g::kMmaWarp) {
    if (c.lane == 0 && c.crank == 0) bf16g::issue<PAIR>(c, w, kp.status);
    __syncwarp();
  } else {
    // drain: exact integer sums of this thread's columns over the segments;
    // only the final sum is reduced mod m
    constexpr int kC = bf16g::kDrainCols;
    const int c0 = (c.warp >> 2) * kC, row = (c.warp & 3) * 32 + c.lane;
    const uint32_t addr = bf16g::drain_addr(c);
    uint32_t seg = 0;
    bool stop = false;
    bf16g::Item t;
    for (int rd = 0; !stop && w.at(rd, c.cid, c.ncl, t); ++rd) {
      const int nseg = (bf16g::stages_of<PAIR>(t) + t.seg - 1) / t.seg;
      const int cols = t.cols - c0;  // of this warp's kC columns
      const int l = t.unit % kp.nm;
      const int p16 = mt.pow16[l][1];
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
          if (q == kC / 16 - 1) bf16g::release_segment<PAIR>(c, seg);
          if (16 * q < cols) {
#pragma unroll
            for (int x = 0; x < 16; ++x) run[16 * q + x] += __float2int_rn(__uint_as_float(v[x]));
          }
        }
        // fold every kFold segments, so that the int32 sums never overflow, whatever K is
        if (s % kFold == kFold - 1) {
#pragma unroll
          for (int x = 0; x < kC; ++x) run[x] = fold16(run[x], p16);
        }
      }
      if (stop) break;
      // Eq. (7): residues in [0, m), kC bytes of this thread's row
      const float m = mt.mf[l], inv = mt.inv[l];
      const float off = __fadd_rn(__fmul_rn(0.5f, inv), -0.5f);
      const int tm = t.tm + static_cast<int>(c.crank);
      uint4* dst = reinterpret_cast<uint4*>(
          kp.R + (static_cast<int64_t>(t.unit) * kp.tiles_m * kBM + tm * kBM + row) * kp.ldr + t.tn * kBN + c0);
#pragma unroll
      for (int g = 0; g < kC / 16; ++g) {
        uint32_t wv[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          int x[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) x[k] = fold16(run[16 * g + 4 * e + k], p16);
          wv[e] = mod4(x, inv, off, -m);
        }
        if (16 * g < cols) dst[g] = make_uint4(wv[0], wv[1], wv[2], wv[3]);
      }
    }
  }
  bf16g::finish<PAIR>(c);
}

// ---------------------------------------------------------------- CRT
constexpr int kCrtCols = 4;  // output columns per thread: one 32-bit word per residue plane

struct KParamsCRT {
  const uint8_t* R;
  int64_t ldr, plane;  // residue row pitch and plane size (bytes)
  int M, N, nm;
  const int32_t* EA;
  const int32_t* FB;
  int escale;
  double alpha_re, alpha_im, beta_re, beta_im;
  void* C;
  int64_t ldc;
  int plain;  // alpha = 1, beta = 0: C = the result (no FP64 update arithmetic)
};

// x of modulus pair i for column c from the interleaved residue bytes:
// t01 = (r, r') of columns 0 and 1, t23 of columns 2 and 3.
__device__ __forceinline__ uint32_t pair_x(uint32_t coef, uint32_t t01, uint32_t t23, int c) {
  const uint32_t t = c < 2 ? t01 : t23;
  return (c & 1) ? __dp2a_hi(coef, t, 0u) : __dp2a_lo(coef, t, 0u);
}

template <int L>
__device__ __forceinline__ void pair_acc(CrtPair<L>& a, const CrtPairTables& ct, int i, uint32_t x) {
#pragma unroll
  for (int j = 0; j < L; ++j) a.s[j] += static_cast<uint64_t>(ct.w[i][j]) * x;
}

// The residue words (four columns each) of one plane set, interleaved by
// pairs of moduli.  All loads are issued first (independent, predicated).
template <int MAXP>
__device__ __forceinline__ void load_pairs(const uint8_t* p, int64_t plane, int nm, uint32_t* t01, uint32_t* t23) {
  uint32_t w[2 * MAXP];
#pragma unroll
  for (int l = 0; l < 2 * MAXP; ++l)
    w[l] = l < nm ? __ldcg(reinterpret_cast<const uint32_t*>(p + static_cast<int64_t>(l) * plane)) : 0u;
#pragma unroll
  for (int i = 0; i < MAXP; ++i) {
    t01[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x5140u);
    t23[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x7362u);
  }
}

// One thread per row and four consecutive columns: the CRT sums of Eq. (8)
// from the residue planes (3M: Re = T1 - T2, Im = T3 - T1 - T2 mod m, Eq.
// 16), S mod P with the symmetric lift, binary64, scaling and the update.
// Bound by integer issue: per output and pair of moduli one dot product of
// two residues with 16-bit coefficients and L wide multiply-adds, half of what
// a weight per modulus took.  n = 8192, 16 moduli: 1.08 -> 0.75 ms (the bytes
// alone take 0.27), 3M 2.80 -> 1.92 ms; 2905 x 1777, 14 moduli: 82 -> 50 us.
// Loops bounded by the 4 L moduli that L limbs hold, not by 20, need 52
// registers instead of 110 at L = 2 (3M, 8 moduli, 3001 x 2047: 115 -> 80 us;
// 16 moduli, n = 8192: 1.92 -> 1.72 ms).
template <int MODE, int L>
__global__ void __launch_bounds__(256) crt_II_kernel(const __grid_constant__ KParamsCRT kp,
                                                     const __grid_constant__ CrtPairTables ct) {
  grid_begin();
  constexpr bool CPLX = MODE == II_Z3M || MODE == II_C3M;
  constexpr int kP = 2 * L;  // P of L limbs has at most 4 L moduli
  const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int ncq = (kp.N + kCrtCols - 1) / kCrtCols;
  if (idx >= static_cast<int64_t>(kp.M) * ncq) return;
  const int row = static_cast<int>(idx / ncq), c0 = static_cast<int>(idx % ncq) * kCrtCols;
  const uint8_t* const p = kp.R + static_cast<int64_t>(row) * kp.ldr + c0;
  const int erow = kp.EA[row] + kp.escale;
  uint32_t a01[kP], a23[kP];
  load_pairs<kP>(p, kp.plane, kp.nm, a01, a23);
  if constexpr (!CPLX) {
#pragma unroll
    for (int c = 0; c < kCrtCols; ++c) {
      const int cidx = c0 + c;
      if (cidx >= kp.N) break;
      CrtPair<L> acc;
#pragma unroll
      for (int j = 0; j < L; ++j) acc.s[j] = 0;
#pragma unroll
      for (int i = 0; i < kP; ++i) {
        if (2 * i >= kp.nm) break;
        pair_acc<L>(acc, ct, i, pair_x(ct.c[i], a01[i], a23[i], c));
      }
      const double xr = scale2_fast(crt_finish_pair<L>(acc, ct), erow + kp.FB[cidx]);
      if (kp.plain) {  // FP64 is slow on this GPU: no multiply by alpha = 1
        if (MODE == II_F64)
          static_cast<double*>(kp.C)[static_cast<int64_t>(row) * kp.ldc + cidx] = xr;
        else
          static_cast<float*>(kp.C)[static_cast<int64_t>(row) * kp.ldc + cidx] = static_cast<float>(xr);
      } else if (MODE == II_F64) {
        double* cp = static_cast<double*>(kp.C) + static_cast<int64_t>(row) * kp.ldc + cidx;
        *cp = blas_update(kp.alpha_re, xr, kp.beta_re, kp.beta_re != 0.0 ? *cp : 0.0);
      } else {
        float* cp = static_cast<float*>(kp.C) + static_cast<int64_t>(row) * kp.ldc + cidx;
        *cp = static_cast<float>(
            blas_update(kp.alpha_re, xr, kp.beta_re, kp.beta_re != 0.0 ? static_cast<double>(*cp) : 0.0));
      }
    }
  } else {
    const int64_t set = static_cast<int64_t>(kp.nm) * kp.plane;
    uint32_t b01[kP], b23[kP], d01[kP], d23[kP];
    load_pairs<kP>(p + set, kp.plane, kp.nm, b01, b23);
    load_pairs<kP>(p + 2 * set, kp.plane, kp.nm, d01, d23);
#pragma unroll
    for (int c = 0; c < kCrtCols; ++c) {
      const int cidx = c0 + c;
      if (cidx >= kp.N) break;
      CrtPair<L> are, aim;
#pragma unroll
      for (int j = 0; j < L; ++j) are.s[j] = aim.s[j] = 0;
#pragma unroll
      for (int i = 0; i < kP; ++i) {
        if (2 * i >= kp.nm) break;
        // T1 - T2 and T3 - T1 - T2 modulo m m', kept non-negative by a
        // multiple of it: the pair's weight times m m' is a multiple of P
        const uint32_t t1 = pair_x(ct.c[i], a01[i], a23[i], c), t2 = pair_x(ct.c[i], b01[i], b23[i], c);
        const uint32_t t3 = pair_x(ct.c[i], d01[i], d23[i], c);
        pair_acc<L>(are, ct, i, t1 + ct.off[i] - t2);
        pair_acc<L>(aim, ct, i, t3 + 2 * ct.off[i] - t1 - t2);
      }
      const int sc = erow + kp.FB[cidx];
      const double xr = scale2_fast(crt_finish_pair<L>(are, ct), sc);
      const double xi = scale2_fast(crt_finish_pair<L>(aim, ct), sc);
      // complex update in binary64; complex64 output rounds each part once more
      using TO = typename std::conditional<MODE == II_C3M, float, double>::type;
      TO* cp = static_cast<TO*>(kp.C) + 2 * (static_cast<int64_t>(row) * kp.ldc + cidx);
      if (kp.plain) {
        cp[0] = static_cast<TO>(xr);
        cp[1] = static_cast<TO>(xi);
        continue;
      }
      double tr = __fma_rn(kp.alpha_re, xr, -__dmul_rn(kp.alpha_im, xi));
      double ti = __fma_rn(kp.alpha_re, xi, __dmul_rn(kp.alpha_im, xr));
      if (kp.beta_re != 0.0 || kp.beta_im != 0.0) {
        const double cr = static_cast<double>(cp[0]), ci = static_cast<double>(cp[1]);
        tr = __dadd_rn(tr, __fma_rn(kp.beta_re, cr, -__dmul_rn(kp.beta_im, ci)));
        ti = __dadd_rn(ti, __fma_rn(kp.beta_re, ci, __dmul_rn(kp.beta_im, cr)));
      }
      cp[0] = static_cast<TO>(tr);
      cp[1] = static_cast<TO>(ti);
    }
  }
}

cudaError_t launch_residues(const GemmIIArgs& a, int nsets, const ModTables& mt, cudaStream_t st) {
  const bool pair = a.cluster == 2;
  KParamsIITC kp;
  kp.tA = *a.descA;
  kp.tB = *a.descB;
  kp.nst = (a.K + 63) / 64;
  kp.tiles_m = (a.M + kBM - 1) / kBM;
  if (pair) kp.tiles_m += kp.tiles_m & 1;  // whole pair tiles: the residue planes hold them
  kp.tiles_n = (a.N + kBN - 1) / kBN;
  kp.N = a.N;
  kp.nplanes = nsets * a.nm;
  kp.nm = a.nm;
  kp.rowsA_pad = a.rowsA_pad;
  kp.rowsB_pad = a.rowsB_pad;
  kp.R = a.scratch;
  kp.ldr = static_cast<int64_t>(kp.tiles_n) * kBN;
  kp.status = a.status;
  const int64_t nitems = static_cast<int64_t>(kp.nplanes) * (pair ? kp.tiles_m / 2 : kp.tiles_m) * kp.tiles_n;
  if (nitems == 0 || kp.nst == 0) return cudaSuccess;
  return pair ? bf16g::launch<true>(gemm_II_tc_kernel<true>, nitems, a.num_sms, st, kp, mt)
              : bf16g::launch<false>(gemm_II_tc_kernel<false>, nitems, a.num_sms, st, kp, mt);
}

template <int MODE>
cudaError_t launch_crt(const GemmIIArgs& a, const CrtPairTables& ct, cudaStream_t st) {
  KParamsCRT kp;
  const int cl = a.cluster;
  const int tiles_m = ((a.M + kBM - 1) / kBM + cl - 1) / cl * cl;
  kp.R = a.scratch;
  kp.ldr = static_cast<int64_t>((a.N + kBN - 1) / kBN) * kBN;
  kp.plane = static_cast<int64_t>(tiles_m) * kBM * kp.ldr;
  kp.M = a.M;
  kp.N = a.N;
  kp.nm = a.nm;
  kp.EA = a.EA;
  kp.FB = a.FB;
  kp.escale = a.escale;
  kp.alpha_re = a.alpha_re;
  kp.alpha_im = a.alpha_im;
  kp.beta_re = a.beta_re;
  kp.beta_im = a.beta_im;
  kp.C = a.C;
  kp.ldc = a.ldc;
  kp.plain = a.alpha_re == 1.0 && a.alpha_im == 0.0 && a.beta_re == 0.0 && a.beta_im == 0.0;
  const int64_t threads = static_cast<int64_t>(a.M) * ((a.N + kCrtCols - 1) / kCrtCols);
  if (threads == 0) return cudaSuccess;
  const unsigned grid = static_cast<unsigned>((threads + 255) / 256);
  switch (ct.limbs) {
    case 2: return launch_after(crt_II_kernel<MODE, 2>, grid, 256, st, kp, ct);
    case 3: return launch_after(crt_II_kernel<MODE, 3>, grid, 256, st, kp, ct);
    case 4: return launch_after(crt_II_kernel<MODE, 4>, grid, 256, st, kp, ct);
    default: return launch_after(crt_II_kernel<MODE, 5>, grid, 256, st, kp, ct);
  }
}

// part: 1 = the residue GEMM, 2 = the CRT kernel, 3 = both.
template <int MODE>
cudaError_t launch_mode(const GemmIIArgs& a, const ModTables& mt, const CrtPairTables& ct, cudaStream_t st, int part) {
  constexpr int NSET = (MODE == II_Z3M || MODE == II_C3M) ? 3 : 1;
  if (part & 1) {
    cudaError_t e = launch_residues(a, NSET, mt, st);
    if (e != cudaSuccess) return e;
  }
  return (part & 2) ? launch_crt<MODE>(a, ct, st) : cudaSuccess;
}

}  // namespace

int gemm_II_tc_tile_m() { return kBM; }
int gemm_II_tc_tile_n() { return kBN; }

size_t gemm_II_tc_residue_bytes(int64_t M, int64_t N, int nm, bool is_complex, int cluster) {
  const int64_t tiles_m = ((M + kBM - 1) / kBM + cluster - 1) / cluster * cluster;
  const int64_t tiles_n = (N + kBN - 1) / kBN;
  return static_cast<size_t>(is_complex ? 3 : 1) * nm * static_cast<size_t>(tiles_m * kBM) *
         static_cast<size_t>(tiles_n * kBN);
}

// Pairs need full 256-row tiles (an odd number of 128-row tiles leaves half a
// pair idle, which costs more than pairs gain below 5) and long segments.
static bool use_pairs(int64_t M, int64_t K) {
  const int64_t t = (M + kBM - 1) / kBM;
  return (t % 2 == 0 || t >= 5) && K >= kPairMinK;
}

// CTAs per GEMM tile of a product of M rows: 2 (a CTA pair on a 256 x 256
// tile) or 1 (128 x 256), or always the one that EMU_II_CLUSTER names.  The B
// tensor map's box is 256 / cluster rows.
int gemm_II_tc_cluster(int64_t M, int64_t K) {
  static int v = -1;
  if (v < 0) {
    const char* e = std::getenv("EMU_II_CLUSTER");
    const int x = e ? std::atoi(e) : 0;
    v = x == 1 || x == 2 ? x : 0;
  }
  return v ? v : use_pairs(M, K) ? 2 : 1;
}

cudaError_t launch_gemm_II_tc(int out_mode, const GemmIIArgs& a, const ModTables& mt, const CrtPairTables& ct,
                              cudaStream_t st, int part) {
  switch (out_mode) {
    case II_F64:
      return launch_mode<II_F64>(a, mt, ct, st, part);
    case II_F32:
      return launch_mode<II_F32>(a, mt, ct, st, part);
    case II_Z3M:
      return launch_mode<II_Z3M>(a, mt, ct, st, part);
    case II_C3M:
      return launch_mode<II_C3M>(a, mt, ct, st, part);
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace emu
