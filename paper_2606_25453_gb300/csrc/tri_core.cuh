// tri_core.cuh -- the digit triangle of Scheme I (Eq. 2) as bf16 products:
// which planes an operand is split into, and which integer products of them
// give the exact partials.
//
// The slices D_t of Eq. (1) (slice 0 in [-128, 127], tails in [0, 255]) are
// recentred: D_t = d_t + 128 e_t with e_0 = 0, e_t = 1, so every d_t lies in
// [-128, 127].  With c(i, j) = sum_k d_i d'_j,
//   S = sum_{i+j<p} 256^(p-1-i-j) sum_k D_i D'_j
//     = sum_s 256^(p-1-s) T_s + R_row + Q_col,   T_s = sum_{i+j=s} c(i, j),
// where R and Q hold the products with the constant 128s and need only the
// sums over k of each operand's digits.
//
// The cross terms of T_s are formed in pairs from ONE product of digit sums
// (Karatsuba): c(i, j) + c(j, i) = x(i, j) - c(i, i) - c(j, j) with
// x(i, j) = sum_k (d_i + d_j)(d'_i + d'_j).  Digit sums lie in [-256, 254]
// and are exact bf16 values.  Used for all i < j except (0, p - 1), whose
// two products are formed directly (c(p-1, p-1) would serve this pair
// alone), the triangle takes 24 products at p = 8 instead of 36, 15 instead
// of 21 at p = 6, 8 instead of 10 at p = 4.  The integers are the same, so S
// is the same.
//
// An FP32 accumulator holds every integer up to 2^24: sums of 1024 digit
// products (2^14 each) or of 256 digit-sum products (2^16 each) are exact.
#pragma once
#include <cstdint>

namespace emu {

// Digit-sum planes: (i, j), i < j, i + j <= p - 1, without (0, p - 1).
constexpr int tri_cross(int p) {
  int n = 0;
  for (int i = 0; i < p; ++i)
    for (int j = i + 1; i + j <= p - 1; ++j) n += !(i == 0 && j == p - 1);
  return n;
}
// Planes of one split operand: p digits, then the digit sums in (i, j) order.
constexpr int tri_planes(int p) { return p + tri_cross(p); }
// Index of digit sum (i, j) among the planes.
constexpr int tri_cross_plane(int p, int i, int j) {
  int n = p;
  for (int a = 0; a < i; ++a)
    for (int b = a + 1; a + b <= p - 1; ++b) n += !(a == 0 && b == p - 1);
  for (int b = i + 1; b < j; ++b) n += !(i == 0 && b == p - 1);
  return n;
}
// Diagonal products c(i, i): i = 0 .. tri_diag(p) - 1.
constexpr int tri_diag(int p) { return p > 1 ? p - 1 : 1; }

constexpr int kTriMaxP = 12;
constexpr int kTriMaxProducts = tri_cross(kTriMaxP) + tri_diag(kTriMaxP) + 2;

// One unit of the triangle: products of plane pairs summed into one int32
// output plane per K chunk.
struct TriUnit {
  uint8_t first, count;  // its plane pairs: pa[first ..], pb[first ..]
  uint8_t sums;          // digit sums (products up to 2^16), else digits (2^14)
  uint8_t out;           // output plane (times the number of K chunks)
};

// Output planes, in this order: per s the units of x(., .) with i + j = s
// (nx[s] of them), then c(i, i), then the direct pair.
struct TriPlan {
  int nunits;
  TriUnit unit[kTriMaxProducts];  // longest first
  uint8_t pa[kTriMaxProducts], pb[kTriMaxProducts];
};

}  // namespace emu
