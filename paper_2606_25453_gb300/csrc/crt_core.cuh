// crt_core.cuh -- multi-word CRT accumulation and finish (Eq. 8 and the
// inverse scaling after it), shared by the Scheme II kernels.
#pragma once
#include "emu_internal.h"

namespace emu {

constexpr int kSL = kCrtLimbs + 1;  // CRT accumulator limbs (S < nm * 256 * P)

// S += w * r for a 5-limb w and r < 256.
__device__ __forceinline__ void crt_acc(uint32_t* S, const uint32_t* w, uint32_t r) {
  uint64_t c = 0;
#pragma unroll
  for (int i = 0; i < kCrtLimbs; ++i) {
    c += static_cast<uint64_t>(w[i]) * r + S[i];
    S[i] = static_cast<uint32_t>(c);
    c >>= 32;
  }
  S[kCrtLimbs] += static_cast<uint32_t>(c);
}

// Round a nonnegative 5-limb integer to binary64, nearest-even.  Below
// 2^128 the four low limbs are rounded directly; otherwise the window of
// limbs 1..4 (>= 97 significant bits) plus a sticky bit for limb 0 has the
// same rounding, scaled back by 2^32 exactly.  Straight-line code: no limb
// is indexed at run time.
__device__ __forceinline__ double limbs_to_double_rn(const uint32_t* x) {
  if (x[4] == 0) {
    const unsigned __int128 u = (static_cast<unsigned __int128>(x[3]) << 96) |
                                (static_cast<unsigned __int128>(x[2]) << 64) |
                                (static_cast<unsigned __int128>(x[1]) << 32) | x[0];
    return u128_to_double_rn(u);
  }
  unsigned __int128 u = (static_cast<unsigned __int128>(x[4]) << 96) |
                        (static_cast<unsigned __int128>(x[3]) << 64) |
                        (static_cast<unsigned __int128>(x[2]) << 32) | x[1];
  if (x[0]) u |= 1;
  return __dmul_rn(u128_to_double_rn(u), 4294967296.0);  // exact power-of-two scaling
}

// Eq. (8) finish: S mod P, symmetric lift, binary64.
__device__ __forceinline__ double crt_finish(const uint32_t* S, const CrtTables& ct) {
  // quotient estimate q = floor(S / P) <= nm * 255, corrected exactly below
  double sd = 0.0;
#pragma unroll
  for (int i = kSL - 1; i >= 0; --i) sd = __fma_rn(sd, 4294967296.0, static_cast<double>(S[i]));
  int q = static_cast<int>(floor(__dmul_rn(sd, ct.invP)));
  if (q < 0) q = 0;
  // R = S - q * P (6 limbs, may go negative by < 2P)
  uint32_t R[kSL];
  {
    uint64_t mul = 0;
    int64_t br = 0;
#pragma unroll
    for (int i = 0; i < kSL; ++i) {
      uint64_t pi = i < kCrtLimbs ? ct.P[i] : 0u;
      mul += pi * static_cast<uint64_t>(q);
      int64_t d = static_cast<int64_t>(S[i]) - static_cast<int64_t>(static_cast<uint32_t>(mul)) - br;
      mul >>= 32;
      br = d < 0;
      R[i] = static_cast<uint32_t>(d + (br ? (1ll << 32) : 0));
    }
  }
  // fix up: while R < 0 add P; while R >= P subtract P (at most a few steps)
  for (int step = 0; step < 4; ++step) {
    if (static_cast<int32_t>(R[kSL - 1]) < 0) {  // negative (two's complement, 6 limbs)
      uint64_t c = 0;
#pragma unroll
      for (int i = 0; i < kSL; ++i) {
        c += static_cast<uint64_t>(R[i]) + (i < kCrtLimbs ? ct.P[i] : 0u);
        R[i] = static_cast<uint32_t>(c);
        c >>= 32;
      }
      continue;
    }
    bool ge = R[kSL - 1] != 0;
    if (!ge) {
      ge = true;
      for (int i = kCrtLimbs - 1; i >= 0; --i) {
        if (R[i] != ct.P[i]) {
          ge = R[i] > ct.P[i];
          break;
        }
      }
    }
    if (!ge) break;
    int64_t br = 0;
#pragma unroll
    for (int i = 0; i < kSL; ++i) {
      int64_t d = static_cast<int64_t>(R[i]) - (i < kCrtLimbs ? ct.P[i] : 0u) - br;
      br = d < 0;
      R[i] = static_cast<uint32_t>(d + (br ? (1ll << 32) : 0));
    }
  }
  // symmetric lift: R > floor(P/2) -> R - P
  bool gt = false;
  for (int i = kCrtLimbs - 1; i >= 0; --i) {
    if (R[i] != ct.Phalf[i]) {
      gt = R[i] > ct.Phalf[i];
      break;
    }
  }
  if (gt) {
    uint32_t mag[kCrtLimbs];
    int64_t br = 0;
#pragma unroll
    for (int i = 0; i < kCrtLimbs; ++i) {
      int64_t d = static_cast<int64_t>(ct.P[i]) - R[i] - br;
      br = d < 0;
      mag[i] = static_cast<uint32_t>(d + (br ? (1ll << 32) : 0));
    }
    return -limbs_to_double_rn(mag);
  }
  return limbs_to_double_rn(R);
}

// ---------------------------------------------------------------- pair form
// S = sum over pairs of moduli of W x, with x the residue modulo m m' of one
// pair (not reduced) and W < P its CRT weight, kept as one 64-bit sum per
// 32-bit limb of W: at most ten x < 2^27, so no carries until the end.  Half
// the multi-word products of a sum over single moduli.
template <int L>
struct CrtPair {
  uint64_t s[L];
};

// Finish: x = S - k P with k = round(S / P) from the top 64 bits of S and a
// 64-bit reciprocal of P (k is exact unless S / P lies within 8 units of its
// fixed-point form from a half, which the exact comparison below settles),
// |x| <= P / 2, rounded once to binary64.  L 32-bit limbs of P.
template <int L>
__device__ __forceinline__ double crt_finish_pair(const CrtPair<L>& a, const CrtPairTables& ct) {
  static_assert(L >= 2 && L <= kCrtLimbs, "limb count");
  uint32_t S[L + 1];
  uint64_t c = 0;
#pragma unroll
  for (int i = 0; i < L; ++i) {
    c += a.s[i] & 0xFFFFFFFFull;  // two 32-bit halves of each 64-bit sum
    S[i] = static_cast<uint32_t>(c);
    c = (c >> 32) + (a.s[i] >> 32);
  }
  S[L] = static_cast<uint32_t>(c);
  // S / 2^e, e = 32 (L - 2) + sh, in 64 bits (S < 2^31 P)
  const uint64_t hi = (static_cast<uint64_t>(S[L]) << 32) | S[L - 1];
  const uint64_t sn = ct.sh == 32 ? hi : (hi << (32 - ct.sh)) | (S[L - 2] >> ct.sh);
  const uint64_t q = __umul64hi(sn, ct.recip);  // (S / P) 2^frac, at most 2 low
  const uint32_t half = 1u << (ct.frac - 1);
  const uint32_t k = static_cast<uint32_t>((q + half) >> ct.frac);
  uint32_t R[L];  // S - k P modulo 2^(32 L), which holds |x| <= P / 2 with its sign
  {
    uint64_t m = 0;
    uint32_t br = 0;
#pragma unroll
    for (int i = 0; i < L; ++i) {
      m += static_cast<uint64_t>(ct.P[i]) * k;
      const uint64_t d = static_cast<uint64_t>(S[i]) - static_cast<uint32_t>(m) - br;
      R[i] = static_cast<uint32_t>(d);
      br = static_cast<uint32_t>(d >> 63);
      m >>= 32;
    }
  }
  bool neg = static_cast<int32_t>(R[L - 1]) < 0;
  const uint32_t f = static_cast<uint32_t>(q) & (2u * half - 1u);
  if (f - (half - 8u) <= 16u) {
    // S / P next to a half: the fraction of k is not certain.  With k as
    // floor(S / P + 1/2) or one off, x lies in (-P, P); lift it into
    // (-P / 2, P / 2] exactly.  (P is below 2^(32 L); the sign of x comes from
    // comparing S with k P over L + 1 limbs.)
    uint64_t m = 0;
    int64_t top = 0;
    uint32_t br = 0;
#pragma unroll
    for (int i = 0; i <= L; ++i) {
      m += i < L ? static_cast<uint64_t>(ct.P[i < L ? i : 0]) * k : 0ull;
      const uint64_t d = static_cast<uint64_t>(S[i]) - static_cast<uint32_t>(m) - br;
      if (i < L) R[i] = static_cast<uint32_t>(d);
      top = static_cast<int64_t>(d);
      br = static_cast<uint32_t>(d >> 63);
      m >>= 32;
    }
    neg = top < 0;
    // |x| against P / 2 by halves: x > P / 2 -> x - P, x <= -P / 2 -> x + P
    uint32_t mag[L];
    uint64_t cy = neg ? 1 : 0;
#pragma unroll
    for (int i = 0; i < L; ++i) {
      cy += neg ? ~R[i] : R[i];
      mag[i] = static_cast<uint32_t>(cy);
      cy >>= 32;
    }
    int cmp = 0;  // sign of mag - P / 2
#pragma unroll
    for (int i = L - 1; i >= 0; --i)
      if (cmp == 0 && mag[i] != ct.Phalf[i]) cmp = mag[i] > ct.Phalf[i] ? 1 : -1;
    if (neg ? cmp >= 0 : cmp > 0) {
      uint32_t b2 = 0;
#pragma unroll
      for (int i = 0; i < L; ++i) {
        const uint64_t d = static_cast<uint64_t>(ct.P[i]) - mag[i] - b2;
        mag[i] = static_cast<uint32_t>(d);
        b2 = static_cast<uint32_t>(d >> 63);
      }
      neg = !neg;
    }
    uint32_t m5[kCrtLimbs] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < L; ++i) m5[i] = mag[i];
    const double v = limbs_to_double_rn(m5);
    return neg ? bitsd(dbits(v) ^ 0x8000000000000000ull) : v;
  }
  uint32_t mag[kCrtLimbs] = {0, 0, 0, 0, 0};
  uint64_t cy = neg ? 1 : 0;
#pragma unroll
  for (int i = 0; i < L; ++i) {
    cy += neg ? ~R[i] : R[i];
    mag[i] = static_cast<uint32_t>(cy);
    cy >>= 32;
  }
  const double v = limbs_to_double_rn(mag);
  return neg ? bitsd(dbits(v) ^ 0x8000000000000000ull) : v;  // sign flip without an FP64 instruction
}

// x 2^e for a nonzero finite x whose result stays normal: exponent-field
// arithmetic (exact, as is ldexp); other cases go to ldexp.
__device__ __forceinline__ double scale2_fast(double x, int e) {
  const uint64_t b = dbits(x);
  const int ex = static_cast<int>((b >> 52) & 0x7FF);
  if (ex == 0 || ex == 0x7FF || ex + e <= 0 || ex + e >= 0x7FF) return ldexp(x, e);
  return bitsd(b + (static_cast<uint64_t>(static_cast<int64_t>(e)) << 52));
}

}  // namespace emu
