// split_tri.cu -- Scheme I split for the bf16 digit triangle (tri_core.cuh):
// the recentred digits d_t of every element and the digit sums d_i + d_j as
// bf16 planes, and the sums of each vector's digits over K.
//
// Planes: plane q, vector r, element h at element (q * rows + r) * kpad + h
// (bf16); kpad is K rounded up to 64, the padding is zero.  Rows are not
// padded: a row of A only reaches the same row of C.
//
// HBM bound: 8 bytes read and 2 per plane written per element (23 planes at
// p = 8).
#include "emu_internal.h"
#include "split_tri_core.cuh"

namespace emu {
namespace {

// K-contiguous source: one warp per (vector, run of `per` groups of 128
// elements); lane l takes elements 4l .. 4l+3 of each group.
template <typename T, int P>
__global__ void __launch_bounds__(256) split_tri_kcontig(const T* __restrict__ X, int64_t ld, int64_t rows, int64_t k,
                                                         int64_t kpad, int per, int64_t nseg,
                                                         const unsigned long long* maxbits,
                                                         uint16_t* __restrict__ planes, int32_t* __restrict__ E_out,
                                                         int32_t* __restrict__ sums, bool vec) {
  grid_begin();
  const int lane = threadIdx.x & 31;
  const int64_t w = static_cast<int64_t>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  if (w >= rows * nseg) return;
  const int64_t r = w / nseg, g0 = (w % nseg) * per;
  const int E = exp_from_maxbits(maxbits, r, rows);
  int sum[P];
#pragma unroll
  for (int t = 0; t < P; ++t) sum[t] = 0;
  for (int64_t g = g0; g < g0 + per; ++g) {
    const int64_t h0 = g * 128 + lane * 4;
    if (h0 >= kpad) break;
    uint64_t bits[4];
    load4_kcontig(X + r * ld, h0, k, true, vec, bits);
    digits4<P>(bits, E, live_count(h0, k), planes + r * kpad + h0, rows * kpad, sum);
  }
  __syncwarp();
  int mine = 0;
#pragma unroll
  for (int t = 0; t < P; ++t) {
    const int s = __reduce_add_sync(0xFFFFFFFFu, sum[t]);
    if (lane == t) mine = s;
  }
  if (lane < P) atomicAdd(sums + lane * rows + r, mine);
  if (g0 == 0 && lane == 0) E_out[r] = E;
}

// K-strided source: a block takes TR vectors x `per` groups of 128 elements
// through a shared-memory tile; warp w packs vectors w, w + 8, ..  The
// exponents are read once per block and one vector is packed at a time, so
// that four blocks fit an SM (two when the compiler interleaved vectors): both
// splits of n = 8192, p = 8 took 1.35 ms before, 1.19 after (bytes: 1.06).
template <typename T, int P, int TR>
__global__ void __launch_bounds__(256, P <= 8 ? 4 : 2) split_tri_kstrided(const T* __restrict__ X, int64_t ld, int64_t rows, int64_t k,
                                                          int64_t kpad, int per,
                                                          const unsigned long long* maxbits,
                                                          uint16_t* __restrict__ planes, int32_t* __restrict__ E_out,
                                                          int32_t* __restrict__ sums, bool vec) {
  grid_begin();
  __shared__ uint64_t tile[TR][133];
  __shared__ int ssum[TR][P], sE[TR];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * TR;
  for (int i = threadIdx.x; i < TR * P; i += 256) (&ssum[0][0])[i] = 0;
  if (threadIdx.x < TR && r0 + threadIdx.x < rows) {
    const int E = exp_from_maxbits(maxbits, r0 + threadIdx.x, rows);
    sE[threadIdx.x] = E;
    if (blockIdx.y == 0) E_out[r0 + threadIdx.x] = E;
  }
  for (int64_t g = static_cast<int64_t>(blockIdx.y) * per; g < (static_cast<int64_t>(blockIdx.y) + 1) * per; ++g) {
    const int64_t hbase = g * 128;
    if (hbase >= kpad) break;
    __syncthreads();  // the previous group is done with the tile
    fill_tile_strided<TR>(tile, X, ld, rows, k, r0, hbase, vec);
    __syncthreads();
    const int64_t h0 = hbase + lane * 4;
#pragma unroll 1
    for (int rl = warp; rl < TR; rl += 8) {
      const int64_t r = r0 + rl;
      if (r >= rows) break;
      int sum[P];
#pragma unroll
      for (int t = 0; t < P; ++t) sum[t] = 0;
      if (h0 < kpad) {
        uint64_t bits[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) bits[q] = tile[rl][q * 33 + lane];
        digits4<P>(bits, sE[rl], live_count(h0, k), planes + r * kpad + h0, rows * kpad, sum);
      }
      __syncwarp();
#pragma unroll
      for (int t = 0; t < P; ++t) {
        const int s = __reduce_add_sync(0xFFFFFFFFu, sum[t]);
        if (lane == t) ssum[rl][t] += s;  // only this warp, this lane touches it
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < TR * P; i += 256) {
    const int rl = i % TR, t = i / TR;
    if (r0 + rl < rows) atomicAdd(sums + t * rows + r0 + rl, ssum[rl][t]);
  }
}

template <typename T, int P>
cudaError_t launch_p(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k, const unsigned long long* maxbits,
              uint16_t* planes, int32_t* E, int32_t* sums, int num_sms, cudaStream_t st) {
  const int64_t kpad = (k + 63) / 64 * 64, ngroups = (kpad + 127) / 128;
  const bool vec = vec16_ok(X, ld);
  // groups per warp (block): up to 8, as long as the grid keeps about eight
  // blocks per SM (fewer atomics on the digit sums, no idle SMs)
  const int64_t units = kcontig ? (rows + 7) / 8 : (rows + 31) / 32;
  int per = 8;
  while (per > 1 && units * ((ngroups + per - 1) / per) < 8 * static_cast<int64_t>(num_sms)) per >>= 1;
  int64_t nseg = (ngroups + per - 1) / per;
  if (kcontig) {
    const int64_t blocks = (rows * nseg + 7) / 8;
    return launch_after(split_tri_kcontig<T, P>, static_cast<unsigned>(blocks), 256, st, X, ld, rows, k, kpad, per, nseg,
                        maxbits, planes, E, sums, vec);
  } else {
    while (nseg > 65535) {
      per *= 2;
      nseg = (ngroups + per - 1) / per;
    }
    // Eight vectors per block (64 contiguous bytes per K row of binary64) while
    // 32 would leave SMs without two blocks: a warp then packs one vector
    // instead of four in turn.  p = 7, whole call: n = 256 25.2 -> 21.1 us, n =
    // 1024 94.4 -> 92.4; with enough blocks the shorter rows only cost.
    const bool small = units * nseg < 2 * static_cast<int64_t>(num_sms);
    const dim3 grid(static_cast<unsigned>(small ? (rows + 7) / 8 : units), static_cast<unsigned>(nseg));
    return launch_after(small ? split_tri_kstrided<T, P, 8> : split_tri_kstrided<T, P, 32>, grid, 256, st, X, ld, rows, k,
                        kpad, per, maxbits, planes, E, sums, vec);
  }
}

}  // namespace

template <typename T>
cudaError_t launch_split_tri(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k, int p,
                      const unsigned long long* maxbits, uint16_t* planes, int32_t* E, int32_t* sums, int num_sms,
                      cudaStream_t st) {
  if (rows == 0 || k == 0) return cudaSuccess;
  if (const cudaError_t e = fault_step(FAULT_SPLIT); e != cudaSuccess) return e;
  switch (p) {
#define EMU_CASE(PP) \
  case PP:           \
    return launch_p<T, PP>(X, ld, kcontig, rows, k, maxbits, planes, E, sums, num_sms, st);
    EMU_CASE(1) EMU_CASE(2) EMU_CASE(3) EMU_CASE(4) EMU_CASE(5) EMU_CASE(6)
    EMU_CASE(7) EMU_CASE(8) EMU_CASE(9) EMU_CASE(10) EMU_CASE(11) EMU_CASE(12)
#undef EMU_CASE
    default:
      return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_split_tri<double>(const double*, int64_t, bool, int64_t, int64_t, int, const unsigned long long*,
                                       uint16_t*, int32_t*, int32_t*, int, cudaStream_t);
template cudaError_t launch_split_tri<float>(const float*, int64_t, bool, int64_t, int64_t, int, const unsigned long long*,
                                      uint16_t*, int32_t*, int32_t*, int, cudaStream_t);

}  // namespace emu
