// split_tri_core.cuh -- per-element digits and digit sums of the bf16 digit
// triangle, shared by the single and the grouped splits.
#pragma once
#include "split_core.cuh"
#include "tri_core.cuh"

namespace emu {

// Four consecutive K elements of one vector (binary64 bits) to their digits
// and digit sums; `live` bit q: element q lies inside K (the planes are zero
// outside).  `dst`: the first element in plane 0; `plane`: plane stride in
// elements.  sum[t] gains the four digits d_t.
template <int P>
__device__ __forceinline__ void digits4(const uint64_t* bits, int E, int nlive, uint16_t* dst, int64_t plane,
                                        int* sum) {
  float f[P][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t b[P];
    slice_digits<P>(bits[q], E, b);
    const bool live = q < nlive;
#pragma unroll
    for (int t = 0; t < P; ++t) {
      // byte + 128 (slice 0, signed) or the byte itself (tails), then - 128:
      // 2^23 + u has u in its low mantissa bits
      const uint32_t u = live ? (t == 0 ? b[t] ^ 0x80u : b[t]) : 128u;
      sum[t] += static_cast<int>(u) - 128;
      f[t][q] = __uint_as_float(0x4B000000u | u) - 8388736.0f;
    }
  }
  // integers of magnitude <= 256 are exact bf16 values: the upper half of
  // the binary32 pattern
  auto put = [&](int q, float a, float b, float c, float d) {
    *reinterpret_cast<uint2*>(dst + static_cast<int64_t>(q) * plane) =
        make_uint2(__byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632u),
                   __byte_perm(__float_as_uint(c), __float_as_uint(d), 0x7632u));
  };
#pragma unroll
  for (int t = 0; t < P; ++t) put(t, f[t][0], f[t][1], f[t][2], f[t][3]);
#pragma unroll
  for (int i = 0; i < P; ++i)
#pragma unroll
    for (int j = i + 1; i + j < P; ++j)
      if (!(i == 0 && j == P - 1))
        put(tri_cross_plane(P, i, j), f[i][0] + f[j][0], f[i][1] + f[j][1], f[i][2] + f[j][2], f[i][3] + f[j][3]);
}

__device__ __forceinline__ int live_count(int64_t h0, int64_t k) {
  return h0 >= k ? 0 : (k - h0 >= 4 ? 4 : static_cast<int>(k - h0));
}

}  // namespace emu
