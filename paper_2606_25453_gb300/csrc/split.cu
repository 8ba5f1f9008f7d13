// split.cu -- exponent scan and slice / residue packing (HBM-bound steps).
//
// Scan (Eq. 1 scale vectors; Scheme II scaling): for every reduction vector
// of an operand (row of A, column of B) the largest |x| is found by an
// unsigned max over the IEEE-754 bit patterns with the sign cleared (which
// orders finite magnitudes), so the scan does no floating-point arithmetic.
// Non-finite values have bit patterns >= 0x7FF0... and set the status word.
//
// Split I (Eq. 1, layout Eq. 11): x = trunc(a * 2^(8p-1-E)) taken exactly
// from the bits of a; the p bytes of the 8p-bit two's complement of x are
// the slices (leading slice signed, tails unsigned), written interleaved:
// row r, K-chunk c (32 wide), slice t at bytes [(c*p+t)*32, +32).
//
// Split I on E4M3 slices: the same layout with beta = 5 balanced base-32
// digits stored as exact E4M3 bytes (the FP8 formulation of Sec. VII).
//
// Split II (Eq. 5): a' = trunc(a * 2^(b-E)), symmetric residues modulo the
// moduli, one plane per modulus; complex input also writes the residues of
// a'_re + a'_im for the 3M product (Eq. 16).
#include "emu_internal.h"
#include "split_core.cuh"

namespace emu {

// ------------------------------------------------------------------ loads
template <typename T>
__device__ __forceinline__ uint64_t load_bits(const T* p);
template <>
__device__ __forceinline__ uint64_t load_bits<double>(const double* p) {
  return dbits(__ldg(p));
}
template <>
__device__ __forceinline__ uint64_t load_bits<float>(const float* p) {
  return dbits(static_cast<double>(__ldg(p)));
}

// ------------------------------------------------------------------ scan
// Vector r, element h of an operand: kcontig -> X[(r*ld + h)*cw + part],
// else X[(h*ld + r)*cw + part]; cw = 2 for complex (both parts scanned).
// seg: elements of a vector per block row (K segment), chosen by the launcher.
// One launch scans both operands of a product (the blocks of the first, then
// those of the second): small products are bound by launches.
template <typename T>
struct ScanOperand {
  const T* X;
  int64_t ld, rows, k, seg;
  int64_t vb, blocks;  // blocks per K segment; all blocks
  unsigned long long* maxbits;
  int cw;
  bool kcontig, vec;  // vec: 16-byte loads (every vector starts on a 16-byte boundary)
};

// Float magnitudes are compared on their own bit patterns and the largest
// is widened once (widening is exact and monotone).
template <typename T>
__device__ __forceinline__ uint64_t widen_absbits(uint64_t b);
template <>
__device__ __forceinline__ uint64_t widen_absbits<double>(uint64_t b) {
  return b;
}
template <>
__device__ __forceinline__ uint64_t widen_absbits<float>(uint64_t b) {
  return dbits(static_cast<double>(__uint_as_float(static_cast<uint32_t>(b))));
}
// |scalar j| of a uint4 as unsigned bits of T's width (sign cleared)
template <typename T>
__device__ __forceinline__ uint64_t lane_absbits(const uint4& v, int j) {
  if constexpr (sizeof(T) == 8) {
    const uint32_t lo = j == 0 ? v.x : v.z, hi = j == 0 ? v.y : v.w;
    return ((static_cast<uint64_t>(hi) << 32) | lo) & 0x7FFFFFFFFFFFFFFFull;
  } else {
    const uint32_t w = j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w;
    return w & 0x7FFFFFFFu;
  }
}

template <typename T>
__device__ __forceinline__ uint64_t scalar_absbits(T x) {
  if constexpr (sizeof(T) == 8)
    return dbits(x) & 0x7FFFFFFFFFFFFFFFull;
  else
    return __float_as_uint(x) & 0x7FFFFFFFu;
}

// K-contiguous: one warp per (vector, segment of seg scalars); with vec lane
// l loads the 16 bytes l, l + 32, ..
template <typename T>
__device__ __forceinline__ void scan_kcontig(const ScanOperand<T>& op, int64_t bx, int64_t by, int* status) {
  constexpr int S = 16 / static_cast<int>(sizeof(T));
  const int lane = threadIdx.x & 31;
  const int64_t r = bx * 8 + (threadIdx.x >> 5);
  if (r >= op.rows) return;
  const int64_t len = op.k * op.cw, h0 = by * op.seg;
  const int64_t h1 = h0 + op.seg < len ? h0 + op.seg : len;
  const T* row = op.X + r * op.ld * op.cw;
  uint64_t mx = 0;
  int64_t h = h0;
  if (op.vec) {
    const int64_t nv = (h1 - h0) / S;
    const uint4* pv = reinterpret_cast<const uint4*>(row + h0);
#pragma unroll 4
    for (int64_t i = lane; i < nv; i += 32) {
      const uint4 v = __ldg(pv + i);
#pragma unroll
      for (int j = 0; j < S; ++j) {
        const uint64_t a = lane_absbits<T>(v, j);
        mx = a > mx ? a : mx;
      }
    }
    h += nv * S;  // the ragged end of the row
  }
#pragma unroll 4
  for (h += lane; h < h1; h += 32) {
    const uint64_t a = scalar_absbits<T>(__ldg(row + h));
    mx = a > mx ? a : mx;
  }
  for (int o = 16; o; o >>= 1) {
    const uint64_t w = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = w > mx ? w : mx;
  }
  if (lane == 0 && h0 < h1) {
    mx = widen_absbits<T>(mx);
    atomicMax(op.maxbits + r, static_cast<unsigned long long>(mx));
    if (mx >= 0x7FF0000000000000ull) set_status(status, ST_NONFINITE);
  }
}

// K-strided: lanes along the vectors (coalesced), eight row groups split a K
// segment.  With vec lane x loads the cv vectors x*cv .. (16 bytes), so a
// block takes 32 cv vectors (512 contiguous bytes per warp and K row), else 32.
template <typename T>
__device__ __forceinline__ void scan_kstrided(const ScanOperand<T>& op, int64_t bx, int64_t by, int* status,
                                              uint64_t (*red)[32 * 4]) {
  constexpr int S = 16 / static_cast<int>(sizeof(T));
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, cw = op.cw;
  const int cv = op.vec ? S / cw : 1;
  const int64_t rb = bx * 32 * cv;
  const int64_t r = rb + static_cast<int64_t>(tx) * cv;
  const int64_t h0 = by * op.seg;
  const int64_t h1 = h0 + op.seg < op.k ? h0 + op.seg : op.k;
  uint64_t mx[4] = {0, 0, 0, 0};
  if (op.vec && r + cv <= op.rows) {
#pragma unroll 4
    for (int64_t h = h0 + ty; h < h1; h += 8) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(op.X + (h * op.ld + r) * cw));
#pragma unroll
      for (int j = 0; j < S; ++j) {  // scalar j belongs to vector j / cw (cw is 1 or 2)
        const uint64_t a = lane_absbits<T>(v, j);
        if (cw == 2)
          mx[j >> 1] = a > mx[j >> 1] ? a : mx[j >> 1];
        else
          mx[j] = a > mx[j] ? a : mx[j];
      }
    }
  } else if (r < op.rows) {  // unaligned, or the last vectors of the operand: scalar loads
#pragma unroll 4
    for (int64_t h = h0 + ty; h < h1; h += 8) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (c < cv && r + c < op.rows) {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            if (q < cw) {
              const uint64_t a = scalar_absbits<T>(__ldg(op.X + (h * op.ld + r + c) * cw + q));
              mx[c] = a > mx[c] ? a : mx[c];
            }
          }
        }
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c)
    if (c < cv) red[ty][tx * cv + c] = mx[c];
  __syncthreads();
  const int t = threadIdx.x;
  if (t < 32 * cv && rb + t < op.rows && h0 < h1) {
    uint64_t m = red[0][t];
    for (int q = 1; q < 8; ++q) m = red[q][t] > m ? red[q][t] : m;
    m = widen_absbits<T>(m);
    atomicMax(op.maxbits + rb + t, static_cast<unsigned long long>(m));
    if (m >= 0x7FF0000000000000ull) set_status(status, ST_NONFINITE);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) scan_kernel(const __grid_constant__ ScanOperand<T> a,
                                                   const __grid_constant__ ScanOperand<T> b, int* status) {
  grid_begin();
  __shared__ uint64_t red[8][32 * 4];
  const bool first = blockIdx.x < a.blocks;
  const ScanOperand<T>& op = first ? a : b;
  const int64_t blk = first ? blockIdx.x : blockIdx.x - a.blocks;
  const int64_t bx = blk % op.vb, by = blk / op.vb;
  if (op.kcontig)
    scan_kcontig(op, bx, by, status);
  else
    scan_kstrided(op, bx, by, status, red);
}

// ------------------------------------------------------------------ norm scan
// Norm-based Scheme II scaling: e_r with ||x_r||_2 < 2^e_r, computed exactly
// so that the value does not depend on the summation order.  With E the
// frexp exponent of the row maximum and y = x 2^-E (|y| < 1), every square
// is rounded UP to an integer number of units 2^-64, the integers are summed
// (order-free, 128 bits), and e = E + ceil((bitlen(S) - 64) / 2).
// The value is below 2^64 (y^2 < 1): M^2 (106 bits at most) shifted right
// by s = -sh >= 1 with a sticky round-up, in 64-bit halves; a left shift
// (sh >= 0) only occurs for rows of subnormal numbers.
__device__ __forceinline__ uint64_t sq_ceil64(uint64_t bits, int Emax) {
  const uint64_t ab = bits & 0x7FFFFFFFFFFFFFFFull;
  if (ab == 0) return 0;
  const int ef = static_cast<int>(ab >> 52);
  uint64_t M = ab & ((uint64_t{1} << 52) - 1);
  int q;  // |x| = M 2^q
  if (ef == 0) {
    q = -1074;
  } else {
    M |= uint64_t{1} << 52;
    q = ef - 1075;
  }
  const uint64_t lo = M * M, hi = __umul64hi(M, M);
  const int sh = 2 * (q - Emax) + 64;
  if (sh >= 0) return lo << sh;  // then M^2 2^sh < 2^64, so hi = 0 and lo << sh is exact
  const int s = -sh;
  if (s >= 128) return 1;
  uint64_t r, sticky;
  if (s >= 64) {
    const int t = s - 64;
    r = hi >> t;
    sticky = lo | (t ? (hi << (64 - t)) : 0ull);
  } else {
    r = (hi << (64 - s)) | (lo >> s);
    sticky = lo << (64 - s);
  }
  return r + (sticky != 0 ? 1ull : 0ull);
}

// Exact 128-bit atomic add on (lo, hi) words.
__device__ __forceinline__ void atomic_add_u128(unsigned long long* acc, unsigned __int128 v) {
  const unsigned long long lo = static_cast<unsigned long long>(v), hi = static_cast<unsigned long long>(v >> 64);
  const unsigned long long old = atomicAdd(acc, lo);
  const unsigned long long carry = (old + lo < old) ? 1ull : 0ull;
  if (hi + carry) atomicAdd(acc + 1, hi + carry);
}

__device__ __forceinline__ unsigned __int128 shfl_add_u128(unsigned __int128 v) {
  for (int o = 16; o; o >>= 1) {
    const unsigned long long lo = __shfl_xor_sync(0xffffffffu, static_cast<unsigned long long>(v), o);
    const unsigned long long hi = __shfl_xor_sync(0xffffffffu, static_cast<unsigned long long>(v >> 64), o);
    v += (static_cast<unsigned __int128>(hi) << 64) | lo;
  }
  return v;
}

// One launch sums both operands, the blocks of the first, then those of the
// second, with the shapes of scan_kernel's scalar loads; acc: 2 words per
// vector, zeroed first.  The splits read the exponent off the sum.  Two
// memsets, two sums and two finishing launches before: 300 x 200 x 300, 14
// moduli, as a graph 39.8 -> 28.5 us; 2905 x 1777 x 803 297 -> 278 us.
template <typename T>
struct NormOperand {
  const T* X;
  int64_t ld, rows, k, seg;
  int64_t vb, blocks;  // blocks per K segment; all blocks
  const unsigned long long* maxbits;
  unsigned long long* acc;
  int cw;
  bool kcontig;
};

template <typename T>
__global__ void __launch_bounds__(256) norm_kernel(const __grid_constant__ NormOperand<T> a,
                                                   const __grid_constant__ NormOperand<T> b) {
  grid_begin();
  __shared__ unsigned __int128 red[8][32];
  const bool first = blockIdx.x < a.blocks;
  const NormOperand<T>& op = first ? a : b;
  const int64_t blk = first ? blockIdx.x : blockIdx.x - a.blocks;
  const int64_t bx = blk % op.vb, by = blk / op.vb;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cw = op.cw;
  const int64_t r = op.kcontig ? bx * 8 + warp : bx * 32 + lane;
  // a zero vector adds nothing; a non-finite one was flagged by the scan
  const uint64_t mb = r < op.rows ? __ldcg(op.maxbits + r) : 0ull;
  const bool live = mb != 0 && mb < 0x7FF0000000000000ull;
  const int Emax = live ? frexp_exp_bits(mb) : 0;
  unsigned __int128 sum = 0;
  if (op.kcontig) {
    if (!live) return;
    const int64_t len = op.k * cw, h0 = by * op.seg;
    const int64_t h1 = h0 + op.seg < len ? h0 + op.seg : len;
    const T* row = op.X + r * op.ld * cw;
#pragma unroll 4
    for (int64_t h = h0 + lane; h < h1; h += 32) sum += sq_ceil64(load_bits(row + h), Emax);
    sum = shfl_add_u128(sum);
    if (lane == 0 && sum) atomic_add_u128(op.acc + 2 * r, sum);
    return;
  }
  if (live) {
    const int64_t h0 = by * op.seg, h1 = h0 + op.seg < op.k ? h0 + op.seg : op.k;
#pragma unroll 4
    for (int64_t h = h0 + warp; h < h1; h += 8) {
      const T* p = op.X + (h * op.ld + r) * cw;
      sum += sq_ceil64(load_bits(p), Emax);
      if (cw == 2) sum += sq_ceil64(load_bits(p + 1), Emax);
    }
  }
  red[warp][lane] = sum;
  __syncthreads();
  if (warp == 0 && live) {
    for (int q = 1; q < 8; ++q) sum += red[q][lane];
    if (sum) atomic_add_u128(op.acc + 2 * r, sum);
  }
}

// Exponent e of vector r with ||x||_2 < 2^e from its sum of squares.
__device__ __forceinline__ int exp_from_norm(const unsigned long long* acc, const unsigned long long* maxbits,
                                             int64_t r, int64_t rows) {
  if (r >= rows) return 0;
  const unsigned long long lo = __ldcg(acc + 2 * r), hi = __ldcg(acc + 2 * r + 1);
  const uint64_t mb = __ldcg(maxbits + r);
  if ((lo | hi) == 0 || mb >= 0x7FF0000000000000ull) return 0;
  const int L = hi ? 128 - __clzll(static_cast<long long>(hi)) : 64 - __clzll(static_cast<long long>(lo));
  const int d = L - 64;
  const int ep = d >= 0 ? (d + 1) / 2 : -((-d) / 2);  // ceil(d / 2)
  return frexp_exp_bits(mb) + ep;
}

// ------------------------------------------------------------------ split I
// K-contiguous source: one warp per (row, group of four 32-wide K-chunks);
// lane l handles h = 4l .. 4l+3 of the group and writes one 4-byte word per
// slice (lanes 8c .. 8c+7 fill the 32-byte block of chunk c).
template <typename T, int P, bool F8>
__global__ void split_I_kcontig(const T* __restrict__ X, int64_t ld, int64_t rows, int64_t k,
                                int64_t rows_pad, int64_t nchunks,
                                const unsigned long long* maxbits,
                                int8_t* __restrict__ hat, int32_t* __restrict__ E_out, bool vec) {
  const int lane = threadIdx.x & 31;
  const int64_t ngroups = (nchunks + 3) / 4;
  const int64_t w = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (w >= rows_pad * ngroups) return;
  const int64_t r = w / ngroups, g = w % ngroups;
  const int64_t c = g * 4 + (lane >> 3);  // chunk of this lane
  if (c >= nchunks) return;
  const int64_t h0 = c * 32 + (lane & 7) * 4;
  const int E = exp_from_maxbits(maxbits, r, rows);
  uint64_t bits[4];
  load4_kcontig(X + (r < rows ? r : 0) * ld, h0, k, r < rows, vec, bits);
  uint32_t word[P];
  pack4<P, F8>(bits, E, word);
  uint8_t* row = reinterpret_cast<uint8_t*>(hat) + r * (nchunks * 32 * P);
#pragma unroll
  for (int t = 0; t < P; ++t)
    *reinterpret_cast<uint32_t*>(row + (c * P + t) * 32 + (lane & 7) * 4) = word[t];
  if (c == 0 && lane == 0 && r < rows && E_out) E_out[r] = E;
}

// K-strided source (element (r, h) at X[h*ld + r]): a block of 256 threads
// takes 32 vectors x 128 K-elements at a time, reads them coalesced along r
// into shared memory, then works like the K-contiguous kernel (warp w:
// vectors w, w+8, w+16, w+24; lane l: elements 4l .. 4l+3).  Element h of a
// vector is kept at column (h mod 4) * 33 + h / 4 and vectors are 133 words
// apart, so both the column-wise fill and the lane-wise reads are free of
// bank conflicts.
template <typename T, int P, bool F8>
__global__ void __launch_bounds__(256) split_I_kstrided(const T* __restrict__ X, int64_t ld, int64_t rows, int64_t k,
                                                        int64_t rows_pad, int64_t nchunks,
                                                        const unsigned long long* maxbits,
                                                        int8_t* __restrict__ hat, int32_t* __restrict__ E_out,
                                                        bool vec) {
  __shared__ uint64_t tile[32][133];
  const int64_t g = blockIdx.x;  // group of 4 chunks
  const int64_t hbase = g * 128;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t c = g * 4 + (lane >> 3);
  for (int64_t r0 = static_cast<int64_t>(blockIdx.y) * 32; r0 < rows_pad;
       r0 += static_cast<int64_t>(gridDim.y) * 32) {
    __syncthreads();  // the previous row block is done with the tile
    fill_tile_strided(tile, X, ld, rows, k, r0, hbase, vec);
    __syncthreads();
    for (int rl = warp; rl < 32; rl += 8) {
      const int64_t r = r0 + rl;
      if (r >= rows_pad || c >= nchunks) continue;
      const int E = exp_from_maxbits(maxbits, r, rows);
      uint64_t bits[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) bits[q] = tile[rl][q * 33 + lane];
      uint32_t word[P];
      pack4<P, F8>(bits, E, word);
      uint8_t* row = reinterpret_cast<uint8_t*>(hat) + r * (nchunks * 32 * P);
#pragma unroll
      for (int t = 0; t < P; ++t)
        *reinterpret_cast<uint32_t*>(row + (c * P + t) * 32 + (lane & 7) * 4) = word[t];
      if (c == 0 && lane == 0 && r < rows && E_out) E_out[r] = E;
    }
  }
}

// ------------------------------------------------------------------ split II
// The 16-bit digits of |a'| = trunc(|a| 2^shift) (|a'| < 2^80, so five
// digits), negated for a negative element: a' = sum_j d_j 2^(16 j).
__device__ __forceinline__ void digits16(uint64_t bits, int shift, int* d) {
  const ScaledInt s = scaled_trunc_bits(bits, shift);
  // s.mag 2^s.lsh = |a'| < 2^80 (the row exponent bounds every element), so s.lsh < 80
  const unsigned __int128 v = static_cast<unsigned __int128>(s.mag) << s.lsh;
  const uint64_t lo = static_cast<uint64_t>(v);
  const uint32_t hi = static_cast<uint32_t>(v >> 64);
  const int sg = (bits >> 63) ? -1 : 1;
  d[0] = sg * static_cast<int>(lo & 0xFFFFu);
  d[1] = sg * static_cast<int>((lo >> 16) & 0xFFFFu);
  d[2] = sg * static_cast<int>((lo >> 32) & 0xFFFFu);
  d[3] = sg * static_cast<int>(lo >> 48);
  d[4] = sg * static_cast<int>(hi & 0xFFFFu);
}

// Symmetric residue of a' modulo m_l from its digits.  t = sum_j d_j c_j
// with c_j the symmetric residue of 2^(16 j) (|c_j| <= 128) satisfies
// |t| <= 65535 (1 + 4 * 128) < 2^25.1.  q = floor(RN(RN(t) / m + off / m)) is
// floor((t + off) / m) or one off (the three roundings move the quotient,
// which is below 2^18, by less than 0.05), so r = t - q m lies in
// [-off - m, 2m - off) and one correction each way puts it in
// [-off, m - 1 - off].
__device__ __forceinline__ int sym_residue(const int* d, const ModTables& mt, int l) {
  int t = d[0];
#pragma unroll
  for (int j = 1; j < kResDigits; ++j) t += d[j] * mt.pow16[l][j];
  const int m = static_cast<int>(mt.mods[l]), off = mt.off[l];
  const int q = __float2int_rd(__fmaf_rn(__int2float_rn(t), mt.inv[l], mt.offinv[l]));
  int r = t - q * m;
  if (r < -off) r += m;
  if (r >= m - off) r -= m;
  return r;
}

// The same in binary32 for the bf16 planes: the ND lowest 14-bit digits of
// |a'|, negated for a negative element (|a'| < 2^b, so ND = ceil(b / 14),
// rounded up to 2, 4 or 6, covers it; six cover 2^84).  Every partial sum of
// t = sum_j d_j c_j is an integer with |t| <= 16383 (1 + 5 * 128) < 2^24, so
// the FMA chain is exact, and sym_residue_f below takes the symmetric
// residue of t on the FP32 pipe without a correction step.
template <int ND>
__device__ __forceinline__ void digits14f(uint64_t bits, int shift, float* d) {
  const ScaledInt s = scaled_trunc_bits(bits, shift);
  // a' = 0 keeps its digits +0 (no sign), so that no residue below comes out
  // as -0 (whose bf16 pattern is not that of the integer 0)
  const uint32_t sg = s.mag != 0 ? static_cast<uint32_t>(bits >> 63) << 31 : 0u;
  uint32_t dg[ND];
  if constexpr (ND <= 4) {  // |a'| < 2^(14 ND) <= 2^56: one 64-bit word holds it
    const uint64_t v = s.lsh < 64 ? s.mag << s.lsh : 0ull;
#pragma unroll
    for (int j = 0; j < ND; ++j) dg[j] = static_cast<uint32_t>(v >> (14 * j)) & 0x3FFFu;
  } else {
    // s.mag 2^s.lsh = |a'| < 2^80 (the row exponent bounds every element), so s.lsh < 80
    const unsigned __int128 v = static_cast<unsigned __int128>(s.mag) << s.lsh;
    const uint64_t lo = static_cast<uint64_t>(v);
    const uint64_t hi = static_cast<uint64_t>(v >> 64);
    dg[0] = static_cast<uint32_t>(lo & 0x3FFFu);
    dg[1] = static_cast<uint32_t>((lo >> 14) & 0x3FFFu);
    dg[2] = static_cast<uint32_t>((lo >> 28) & 0x3FFFu);
    dg[3] = static_cast<uint32_t>((lo >> 42) & 0x3FFFu);
    dg[4] = static_cast<uint32_t>(((lo >> 56) | (hi << 8)) & 0x3FFFu);
    dg[5] = static_cast<uint32_t>((hi >> 6) & 0x3FFFu);
  }
#pragma unroll
  for (int j = 0; j < ND; ++j)  // 2^23 + d has d in its low mantissa bits; the sign by bit
    d[j] = __uint_as_float(__float_as_uint(__uint_as_float(0x4B000000u | dg[j]) - 8388608.0f) | sg);
}

// The quotient needs no correction: with c = RN((off + 1/2) / m) and
// inv = RN(1/m), floor(t inv + c) (the exact value; the FMA rounds it
// downward, which never crosses the integer below it) equals
// floor((t + off) / m) for every integer |t| <= 16383 (1 + sum_j>=1 |c_j|)
// -- the range of t for the digit count ND <= 6 -- and every modulus of the
// list.  The half in the offset puts (t + off + 1/2) / m at least 1/(2m)
// from the integers, and the roundings of inv and c move t inv + c by at
// most |t| 2^-32 + 2^-25, below 1/(2m) for ND <= 4 (|t| < 2^22.6); the
// claim is checked exhaustively over the whole range, ND = 6 included, by
// the host tests.
// So r = t - q m is the symmetric residue in [-off, m - 1 - off] at once.
// No step produces -0 from the +0 digits of a' = 0 (t = +0, q = 0).
template <int ND>
__device__ __forceinline__ float sym_residue_f(const float* d, const ModTables& mt, int l) {
  float t = d[0];
#pragma unroll
  for (int j = 1; j < ND; ++j) t = __fmaf_rn(d[j], mt.pow14f[l][j], t);
  const float q = floorf(__fmaf_rd(t, mt.inv[l], mt.offhinv[l]));
  return __fmaf_rn(-q, mt.mf[l], t);
}

__device__ __forceinline__ uint32_t pack_bytes(int r0, int r1, int r2, int r3) {
  const uint32_t lo = __byte_perm(static_cast<uint32_t>(r0), static_cast<uint32_t>(r1), 0x0040u);
  const uint32_t hi = __byte_perm(static_cast<uint32_t>(r2), static_cast<uint32_t>(r3), 0x0040u);
  return __byte_perm(lo, hi, 0x5410u);
}

// Four residues as bf16 (exact: |r| <= 128 has at most 8 significant bits,
// so the upper half of the binary32 value is the bf16 value).
__device__ __forceinline__ uint2 pack_bf16(int r0, int r1, int r2, int r3) {
  const uint32_t f0 = __float_as_uint(__int2float_rn(r0)), f1 = __float_as_uint(__int2float_rn(r1));
  const uint32_t f2 = __float_as_uint(__int2float_rn(r2)), f3 = __float_as_uint(__int2float_rn(r3));
  return make_uint2(__byte_perm(f0, f1, 0x7632u), __byte_perm(f2, f3, 0x7632u));
}

template <bool BF>
__device__ __forceinline__ void store4(int8_t* p, int r0, int r1, int r2, int r3) {
  if (BF)
    *reinterpret_cast<uint2*>(p) = pack_bf16(r0, r1, r2, r3);
  else
    *reinterpret_cast<uint32_t*>(p) = pack_bytes(r0, r1, r2, r3);
}

// The residues of four consecutive K elements of one vector, one store per
// plane (INT8: four bytes, byte q = element q; BF: four bf16 values): real
// (cw = 1) one plane per modulus; complex three (re, im, re + im).
// `re`/`im` hold the binary64 bits of the elements; `base` is the address
// of the first element in plane 0, `plane` the plane stride in bytes.  The
// modulus loop is unrolled so that the table entries are kernel-parameter
// operands.
// Four binary32 residues (integers |r| <= 128, never -0) as bf16.
__device__ __forceinline__ void store4f(int8_t* p, float r0, float r1, float r2, float r3) {
  const uint32_t f0 = __float_as_uint(r0), f1 = __float_as_uint(r1);
  const uint32_t f2 = __float_as_uint(r2), f3 = __float_as_uint(r3);
  *reinterpret_cast<uint2*>(p) = make_uint2(__byte_perm(f0, f1, 0x7632u), __byte_perm(f2, f3, 0x7632u));
}

template <int CW, bool BF, int ND>
__device__ __forceinline__ void residues4(const ModTables& mt, int nm, int shift, const uint64_t* re,
                                          const uint64_t* im, int64_t plane, int8_t* base) {
  if constexpr (BF) {  // bf16 planes: the binary32 form
    float dr[4][ND], di[CW == 2 ? 4 : 1][ND];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      digits14f<ND>(re[q], shift, dr[q]);
      if (CW == 2) digits14f<ND>(im[q], shift, di[q]);
    }
#pragma unroll
    for (int l = 0; l < kMaxModuli; ++l) {
      if (l >= nm) break;
      float rr[4], ri[4], rs[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        rr[q] = sym_residue_f<ND>(dr[q], mt, l);
        if (CW == 2) {
          ri[q] = sym_residue_f<ND>(di[q], mt, l);
          const float m = mt.mf[l], off = mt.offf[l];
          float v = rr[q] + ri[q];
          if (v < -off) v += m;
          if (v >= m - off) v -= m;
          rs[q] = v;
        }
      }
      store4f(base + static_cast<int64_t>(l) * plane, rr[0], rr[1], rr[2], rr[3]);
      if (CW == 2) {
        store4f(base + static_cast<int64_t>(nm + l) * plane, ri[0], ri[1], ri[2], ri[3]);
        store4f(base + static_cast<int64_t>(2 * nm + l) * plane, rs[0], rs[1], rs[2], rs[3]);
      }
    }
  } else {
    int dr[4][kResDigits], di[4][kResDigits];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      digits16(re[q], shift, dr[q]);
      if (CW == 2) digits16(im[q], shift, di[q]);
    }
#pragma unroll
    for (int l = 0; l < kMaxModuli; ++l) {
      if (l >= nm) break;
      int rr[4], ri[4], rs[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        rr[q] = sym_residue(dr[q], mt, l);
        if (CW == 2) {
          ri[q] = sym_residue(di[q], mt, l);
          const int m = static_cast<int>(mt.mods[l]), off = mt.off[l];
          int v = rr[q] + ri[q];
          if (v < -off) v += m;
          if (v >= m - off) v -= m;
          rs[q] = v;
        }
      }
      store4<BF>(base + static_cast<int64_t>(l) * plane, rr[0], rr[1], rr[2], rr[3]);
      if (CW == 2) {
        store4<BF>(base + static_cast<int64_t>(nm + l) * plane, ri[0], ri[1], ri[2], ri[3]);
        store4<BF>(base + static_cast<int64_t>(2 * nm + l) * plane, rs[0], rs[1], rs[2], rs[3]);
      }
    }
  }
}

// Scheme II split.  Planes: set q, modulus l at element
// ((q*nm + l)*rows_pad + r)*kpad + h of `res` (set = 0 for real; 0, 1, 2 =
// re, im, re + im for complex); elements are INT8, or bf16 (BF) for the
// tcgen05 kernel.  Row exponent: of the maximum (worst-case
// scaling) or of the 2-norm (acc).  K-contiguous sources: one warp per
// (vector, 128 K-elements), lane l takes elements 4l .. 4l+3 and writes one
// word per plane; strided sources go through a shared-memory tile of 32
// vectors (16 for complex) x 128 elements as in the Scheme I split.
template <typename T, int CW, bool BF, int ND>
__global__ void split_II_kcontig(const T* __restrict__ X, int64_t ld, int64_t rows, int64_t k, int64_t rows_pad,
                                 int64_t kpad, int nm, int b, const __grid_constant__ ModTables mt,
                                 const unsigned long long* maxbits, const unsigned long long* acc,
                                 int8_t* __restrict__ res, int32_t* __restrict__ E_out, bool vec) {
  grid_begin();
  const int lane = threadIdx.x & 31;
  const int64_t ngroups = kpad / 128;
  const int64_t w = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (w >= rows_pad * ngroups) return;
  const int64_t r = w / ngroups, h0 = (w % ngroups) * 128 + lane * 4;
  const int E = acc ? exp_from_norm(acc, maxbits, r, rows) : exp_from_maxbits(maxbits, r, rows);
  uint64_t re[4], im[4];
  if constexpr (CW == 1) {
    load4_kcontig(X + (r < rows ? r : 0) * ld, h0, k, r < rows, vec, re);
#pragma unroll
    for (int q = 0; q < 4; ++q) im[q] = 0ull;
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const bool valid = r < rows && h0 + q < k;
      const T* p = X + (r * ld + h0 + q) * CW;
      re[q] = valid ? load_bits(p) : 0ull;
      im[q] = valid ? load_bits(p + 1) : 0ull;
    }
  }
  residues4<CW, BF, ND>(mt, nm, b - E, re, im, rows_pad * kpad * (BF ? 2 : 1), res + (r * kpad + h0) * (BF ? 2 : 1));
  if (h0 == 0 && r < rows && E_out) E_out[r] = E;
}

template <typename T, int CW, bool BF, int ND, bool SMALL>
__global__ void __launch_bounds__(256) split_II_kstrided(const T* __restrict__ X, int64_t ld, int64_t rows, int64_t k,
                                                         int64_t rows_pad, int64_t kpad, int nm, int b,
                                                         const __grid_constant__ ModTables mt,
                                                         const unsigned long long* maxbits,
                                                         const unsigned long long* acc, int8_t* __restrict__ res,
                                                         int32_t* __restrict__ E_out, bool vec) {
  grid_begin();
  constexpr int TR = SMALL ? 8 : CW == 2 ? 16 : 32;  // vectors per tile (two tiles for complex)
  __shared__ uint64_t tre[TR][133];
  __shared__ uint64_t tim[CW == 2 ? TR : 1][CW == 2 ? 133 : 1];
  const int64_t hbase = static_cast<int64_t>(blockIdx.x) * 128;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t r0 = static_cast<int64_t>(blockIdx.y) * TR; r0 < rows_pad;
       r0 += static_cast<int64_t>(gridDim.y) * TR) {
    __syncthreads();  // the previous row block is done with the tiles
    if constexpr (CW == 1) {
      fill_tile_strided<TR>(tre, X, ld, rows, k, r0, hbase, vec);
    } else {
      for (int i = threadIdx.x; i < TR * 128; i += 256) {
        const int rl = i % TR, hl = i / TR;
        const int64_t r = r0 + rl, h = hbase + hl;
        const bool valid = r < rows && h < k;
        const T* p = X + (h * ld + r) * CW;
        const int col = (hl & 3) * 33 + (hl >> 2);
        tre[rl][col] = valid ? load_bits(p) : 0ull;
        tim[rl][col] = valid ? load_bits(p + 1) : 0ull;
      }
    }
    __syncthreads();
    for (int rl = warp; rl < TR; rl += 8) {
      const int64_t r = r0 + rl;
      if (r >= rows_pad) continue;
      const int E = acc ? exp_from_norm(acc, maxbits, r, rows) : exp_from_maxbits(maxbits, r, rows);
      uint64_t re[4], im[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        re[q] = tre[rl][q * 33 + lane];
        im[q] = CW == 2 ? tim[rl][q * 33 + lane] : 0ull;
      }
      const int64_t h0 = hbase + lane * 4;
      residues4<CW, BF, ND>(mt, nm, b - E, re, im, rows_pad * kpad * (BF ? 2 : 1), res + (r * kpad + h0) * (BF ? 2 : 1));
      if (h0 == 0 && r < rows && E_out) E_out[r] = E;
    }
  }
}

// ------------------------------------------------------------------ launchers
// K segment (elements of a vector per block) of the scan and norm kernels:
// `seg0` (2048 along K-contiguous rows, 256 down strided columns), halved
// while the grid would hold fewer than four blocks per SM -- small operands
// then still have enough loads in flight -- down to `seg_min`, and doubled
// while the segment count exceeds the grid's y limit.
static int64_t scan_seg(int64_t vec_blocks, int64_t len, int64_t seg0, int64_t seg_min) {
  constexpr int64_t kSms = 152;  // of a GB300
  int64_t seg = seg0;
  while (seg > seg_min && vec_blocks * ((len + seg - 1) / seg) < 4 * kSms) seg >>= 1;
  while ((len + seg - 1) / seg > 65535) seg <<= 1;
  return seg;
}

__global__ void zero_kernel(uint4* p, int64_t n) {
  grid_begin();
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) p[i] = make_uint4(0, 0, 0, 0);
}

cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t st) {
  if (const cudaError_t e = fault_step(FAULT_ZERO); e != cudaSuccess) return e;
  const int64_t n = static_cast<int64_t>((bytes + 15) / 16);
  if (n == 0) return cudaSuccess;
  return launch_after(zero_kernel, static_cast<unsigned>((n + 255) / 256), 256, st, static_cast<uint4*>(p), n);
}

template <typename T>
static ScanOperand<T> scan_operand(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k, int cw,
                                   unsigned long long* maxbits) {
  ScanOperand<T> op{X, ld, rows, k, 0, 1, 0, maxbits, cw, kcontig, false};
  if (rows == 0 || k == 0) return op;
  op.vec = (reinterpret_cast<uintptr_t>(X) & 15u) == 0 && (static_cast<uint64_t>(ld) * cw * sizeof(T)) % 16 == 0;
  const int64_t len = kcontig ? k * cw : k;
  const int64_t per_block = kcontig ? 8 : op.vec ? 32 * static_cast<int64_t>(16 / sizeof(T)) / cw : 32;
  op.vb = (rows + per_block - 1) / per_block;
  op.seg = kcontig ? scan_seg(op.vb, len, 2048, 256) : scan_seg(op.vb, len, 256, 32);
  op.blocks = op.vb * ((len + op.seg - 1) / op.seg);
  return op;
}

template <typename T>
cudaError_t launch_scan(const T* A, int64_t ldA, bool a_kcontig, int64_t M, unsigned long long* maxA, const T* B,
                 int64_t ldB, bool b_kcontig, int64_t N, unsigned long long* maxB, int64_t k, int cw, bool zeroed,
                 int* status, cudaStream_t st) {
  cudaError_t e = fault_step(FAULT_SCAN);
  if (!zeroed) {
    if (e == cudaSuccess && maxA) e = cudaMemsetAsync(maxA, 0, sizeof(*maxA) * M, st);
    if (e == cudaSuccess && maxB) e = cudaMemsetAsync(maxB, 0, sizeof(*maxB) * N, st);
  }
  if (e != cudaSuccess) return e;
  const ScanOperand<T> a = scan_operand(A, ldA, a_kcontig, maxA ? M : 0, k, cw, maxA);
  const ScanOperand<T> b = scan_operand(B, ldB, b_kcontig, maxB ? N : 0, k, cw, maxB);
  if (a.blocks + b.blocks == 0) return cudaSuccess;
  return launch_after(scan_kernel<T>, static_cast<unsigned>(a.blocks + b.blocks), 256, st, a, b, status);
}
template cudaError_t launch_scan<double>(const double*, int64_t, bool, int64_t, unsigned long long*, const double*, int64_t,
                                  bool, int64_t, unsigned long long*, int64_t, int, bool, int*, cudaStream_t);
template cudaError_t launch_scan<float>(const float*, int64_t, bool, int64_t, unsigned long long*, const float*, int64_t,
                                 bool, int64_t, unsigned long long*, int64_t, int, bool, int*, cudaStream_t);

template <typename T, int P, bool F8>
static cudaError_t launch_split_I_p(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k,
                             const unsigned long long* maxbits, int8_t* hat, int32_t* E,
                             cudaStream_t st) {
  int64_t rows_pad = split_rows(rows), nchunks = split_cols_I(k, 1) / 32;
  if (rows_pad == 0 || nchunks == 0) return cudaSuccess;
  if (kcontig) {
    int64_t warps = rows_pad * ((nchunks + 3) / 4);
    int64_t blocks = (warps + 7) / 8;
    split_I_kcontig<T, P, F8><<<static_cast<unsigned>(blocks), 256, 0, st>>>(X, ld, rows, k, rows_pad,
                                                                             nchunks, maxbits, hat, E,
                                                                             vec16_ok(X, ld));
  } else {
    const int64_t rb = rows_pad / 32;
    dim3 grid(static_cast<unsigned>((nchunks + 3) / 4), static_cast<unsigned>(rb < 65535 ? rb : 65535));
    split_I_kstrided<T, P, F8><<<grid, 256, 0, st>>>(X, ld, rows, k, rows_pad, nchunks, maxbits, hat, E,
                                                     vec16_ok(X, ld));
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_split_I(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k, int p,
                    const unsigned long long* maxbits, int8_t* hat, int32_t* E, cudaStream_t st, bool f8) {
  if (const cudaError_t e = fault_step(FAULT_SPLIT); e != cudaSuccess) return e;
  switch (p) {
#define EMU_CASE(PP)                                                                         \
  case PP:                                                                                   \
    return f8 ? launch_split_I_p<T, PP, true>(X, ld, kcontig, rows, k, maxbits, hat, E, st)  \
              : launch_split_I_p<T, PP, false>(X, ld, kcontig, rows, k, maxbits, hat, E, st);
    EMU_CASE(1) EMU_CASE(2) EMU_CASE(3) EMU_CASE(4) EMU_CASE(5) EMU_CASE(6)
    EMU_CASE(7) EMU_CASE(8) EMU_CASE(9) EMU_CASE(10) EMU_CASE(11) EMU_CASE(12)
#undef EMU_CASE
    default:
      return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_split_I<double>(const double*, int64_t, bool, int64_t, int64_t, int,
                                     const unsigned long long*, int8_t*, int32_t*, cudaStream_t, bool);
template cudaError_t launch_split_I<float>(const float*, int64_t, bool, int64_t, int64_t, int,
                                    const unsigned long long*, int8_t*, int32_t*, cudaStream_t, bool);

template <typename T>
cudaError_t launch_split_II(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k, int nm, int b,
                     int cw, const ModTables& tabs, const unsigned long long* maxbits, int8_t* res,
                     int32_t* E, cudaStream_t st, const unsigned long long* acc, bool bf16) {
  const int64_t rows_pad = split_rows(rows), kpad = split_cols_II(k);
  if (rows_pad == 0 || kpad == 0) return cudaSuccess;
  if (const cudaError_t e = fault_step(FAULT_SPLIT); e != cudaSuccess) return e;
  // 14-bit digits that hold |a'| < 2^b (bf16 planes; the INT8 form has its own)
  const int nd = b <= 28 ? 2 : b <= 56 ? 4 : 6;
  const bool vec = cw == 1 && vec16_ok(X, ld);
#define EMU_SPLIT_II_ARGS X, ld, rows, k, rows_pad, kpad, nm, b, tabs, maxbits, acc, res, E, vec
#define EMU_SPLIT_II(KERNEL, GRID, CW)                                             \
  (!bf16     ? launch_after(KERNEL<T, CW, false, 6>, GRID, 256, st, EMU_SPLIT_II_ARGS) \
   : nd == 2 ? launch_after(KERNEL<T, CW, true, 2>, GRID, 256, st, EMU_SPLIT_II_ARGS)  \
   : nd == 4 ? launch_after(KERNEL<T, CW, true, 4>, GRID, 256, st, EMU_SPLIT_II_ARGS)  \
             : launch_after(KERNEL<T, CW, true, 6>, GRID, 256, st, EMU_SPLIT_II_ARGS))
  if (kcontig) {
    const int64_t warps = rows_pad * (kpad / 128);
    const unsigned blocks = static_cast<unsigned>((warps + 7) / 8);
    return cw == 2 ? EMU_SPLIT_II(split_II_kcontig, blocks, 2) : EMU_SPLIT_II(split_II_kcontig, blocks, 1);
  } else {
    // Eight vectors per block while more would leave SMs without a block: a
    // warp then packs one vector instead of two or four in turn.  14 moduli,
    // whole call: n = 512 32.9 -> 27.9 us; n = 1000 (256 blocks of 32) was 73.6
    // and took 74.6 with 8, so the line lies at one block per SM.
    const bool small = bf16 && rows_pad / (cw == 2 ? 16 : 32) * (kpad / 128) < 152;
    const int64_t rb = rows_pad / (small ? 8 : cw == 2 ? 16 : 32);
    dim3 grid(static_cast<unsigned>(kpad / 128), static_cast<unsigned>(rb < 65535 ? rb : 65535));
#define EMU_STRIDED(CW, ND, SMALL) launch_after(split_II_kstrided<T, CW, true, ND, SMALL>, grid, 256, st, EMU_SPLIT_II_ARGS)
#define EMU_STRIDED_ND(CW, SMALL) \
  (nd == 2 ? EMU_STRIDED(CW, 2, SMALL) : nd == 4 ? EMU_STRIDED(CW, 4, SMALL) : EMU_STRIDED(CW, 6, SMALL))
    if (!bf16)
      return cw == 2 ? launch_after(split_II_kstrided<T, 2, false, 6, false>, grid, 256, st, EMU_SPLIT_II_ARGS)
                     : launch_after(split_II_kstrided<T, 1, false, 6, false>, grid, 256, st, EMU_SPLIT_II_ARGS);
    if (cw == 2) return small ? EMU_STRIDED_ND(2, true) : EMU_STRIDED_ND(2, false);
    return small ? EMU_STRIDED_ND(1, true) : EMU_STRIDED_ND(1, false);
#undef EMU_STRIDED_ND
#undef EMU_STRIDED
  }
#undef EMU_SPLIT_II
#undef EMU_SPLIT_II_ARGS
}

template <typename T>
static NormOperand<T> norm_operand(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k, int cw,
                                   const unsigned long long* maxbits, unsigned long long* acc) {
  NormOperand<T> op{X, ld, rows, k, 0, 1, 0, maxbits, acc, cw, kcontig};
  if (rows == 0 || k == 0) return op;
  const int64_t len = kcontig ? k * cw : k;
  op.vb = (rows + (kcontig ? 7 : 31)) / (kcontig ? 8 : 32);
  op.seg = kcontig ? scan_seg(op.vb, len, 2048, 256) : scan_seg(op.vb, len, 256, 32);
  op.blocks = op.vb * ((len + op.seg - 1) / op.seg);
  return op;
}

template <typename T>
cudaError_t launch_norm(const T* A, int64_t ldA, bool a_kcontig, int64_t M, const unsigned long long* maxA,
                 unsigned long long* accA, const T* B, int64_t ldB, bool b_kcontig, int64_t N,
                 const unsigned long long* maxB, unsigned long long* accB, int64_t k, int cw, cudaStream_t st) {
  if (const cudaError_t e = fault_step(FAULT_NORM); e != cudaSuccess) return e;
  const NormOperand<T> a = norm_operand(A, ldA, a_kcontig, accA ? M : 0, k, cw, maxA, accA);
  const NormOperand<T> b = norm_operand(B, ldB, b_kcontig, accB ? N : 0, k, cw, maxB, accB);
  if (a.blocks + b.blocks == 0) return cudaSuccess;
  return launch_after(norm_kernel<T>, static_cast<unsigned>(a.blocks + b.blocks), 256, st, a, b);
}
template cudaError_t launch_norm<double>(const double*, int64_t, bool, int64_t, const unsigned long long*, unsigned long long*,
                                  const double*, int64_t, bool, int64_t, const unsigned long long*,
                                  unsigned long long*, int64_t, int, cudaStream_t);
template cudaError_t launch_norm<float>(const float*, int64_t, bool, int64_t, const unsigned long long*, unsigned long long*,
                                 const float*, int64_t, bool, int64_t, const unsigned long long*, unsigned long long*,
                                 int64_t, int, cudaStream_t);

template cudaError_t launch_split_II<double>(const double*, int64_t, bool, int64_t, int64_t, int, int, int,
                                      const ModTables&, const unsigned long long*, int8_t*, int32_t*,
                                      cudaStream_t, const unsigned long long*, bool);
template cudaError_t launch_split_II<float>(const float*, int64_t, bool, int64_t, int64_t, int, int, int,
                                     const ModTables&, const unsigned long long*, int8_t*, int32_t*,
                                     cudaStream_t, const unsigned long long*, bool);

}  // namespace emu
