// emu_internal.h -- declarations shared by the library's translation units
// (host launchers, layout helpers, method tables passed to kernels).
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "emu_device.cuh"

namespace emu {

// Launch a kernel that begins with grid_begin() so that its launch and the end
// of the kernel before it overlap: a small product is six or seven short
// kernels, and what passed between them was a third of its time.  256^3, p = 7:
// 32.8 -> 22 to 25 us per call (two modes of the host's launch rate); 2905 x
// 1777 x 803, 14 moduli, norm scaling: 278 -> 260; 3001 x 2047 x 2500 complex64:
// 755 -> 742.
template <class... P, class... A>
inline cudaError_t launch_after(void (*kernel)(P...), dim3 grid, unsigned block, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

constexpr int kMaxModuli = 20;  // Scheme II moduli supported
constexpr int kCrtLimbs = 5;     // P < 2^160 for up to 20 moduli
constexpr int kSplitRowAlign = 128;

// Layout of split outputs (see the C ABI header).
inline int64_t split_rows(int64_t rows) { return (rows + kSplitRowAlign - 1) / kSplitRowAlign * kSplitRowAlign; }
inline int64_t split_cols_I(int64_t k, int p) { return (k + 31) / 32 * 32 * p; }
inline int64_t split_cols_II(int64_t k) { return (k + 127) / 128 * 128; }

// Scheme II tables, passed by value to kernels.
// Residues of the scaled integers a' (|a'| < 2^80) are taken from their
// 16-bit digits: a' = sum_j d_j 2^(16 j), a' mod m = sum_j d_j (2^(16 j) mod m)
// mod m, the last reduction in single precision (the sum stays below 2^26).
constexpr int kResDigits = 5;
constexpr int kResDigitsF = 6;
struct ModTables {
  uint32_t mods[kMaxModuli];
  int32_t off[kMaxModuli];                 // m - 1 - floor((m - 1)/2): symmetric residues lie in [-off, m - 1 - off]
  float inv[kMaxModuli];                   // 1/m rounded to nearest
  float offinv[kMaxModuli];                // off/m rounded to nearest
  float offhinv[kMaxModuli];               // (off + 1/2)/m rounded to nearest
  int32_t pow16[kMaxModuli][kResDigits];   // symmetric residue of 2^(16 j) mod m
  // binary32 form for the bf16 planes: 14-bit digits (six cover 2^84)
  float pow14f[kMaxModuli][kResDigitsF];   // symmetric residue of 2^(14 j) mod m
  float mf[kMaxModuli], offf[kMaxModuli];  // m and off as binary32
};

// CRT tables of Eq. (8) for a given number of moduli.
struct CrtTables {
  uint32_t w[kMaxModuli][kCrtLimbs];  // (P/m_l) * q_l, little-endian 32-bit limbs
  uint32_t P[kCrtLimbs];
  uint32_t Phalf[kCrtLimbs];          // floor(P/2)
  double invP;                        // 1/P rounded (quotient estimate only)
  int nm;
};

// The same by pairs of moduli (2 i, 2 i + 1) for crt_finish_pair.
constexpr int kMaxPairs = kMaxModuli / 2;
struct CrtPairTables {
  uint32_t c[kMaxPairs];              // x = r c_lo + r' c_hi is congruent to both residues: 16-bit halves c_lo | c_hi << 16
  uint32_t off[kMaxPairs];            // a multiple of m m' above any x
  uint32_t w[kMaxPairs][kCrtLimbs];   // (P / (m m')) times its inverse modulo m m'
  uint32_t P[kCrtLimbs], Phalf[kCrtLimbs];
  uint64_t recip;                     // floor(2^(63 + bitlen(P)) / P)
  int sh;                             // S is shifted right by e = max(0, bitlen(P) - 32) = 32 (limbs - 2) + sh
  int frac;                           // fraction bits of (S / 2^e) recip / 2^64
  int limbs, nm;                      // 32-bit limbs of P (at least 2)
};

// Host-side method constants (api.cu).
int host_moduli(int nm, int32_t* out);
int64_t host_chunk_len_I(int p);
int64_t host_chunk_len_F8(int p);
int host_scale_bits_II(int nm, int64_t k, int is_complex);
void host_mod_tables(int nm, ModTables* t);
void host_crt_tables(int nm, CrtTables* t);
void host_crt_pair_tables(int nm, CrtPairTables* t);
// The tables of nm moduli, built once per process.
struct MethodTables {
  ModTables mod;
  CrtTables crt;
  CrtPairTables pair;
};
const MethodTables& method_tables(int nm);

// Host-side fault injection (EMU_FAULT, api.cu): the error with which a
// launch of this step fails in place of running, normally none.
enum FaultStep : int { FAULT_ALLOC = 1, FAULT_GEMM, FAULT_ZERO, FAULT_SCAN, FAULT_NORM, FAULT_SPLIT };
cudaError_t fault_step(FaultStep step);

// ---------------------------------------------------------------- launchers
// Each returns its own launch error: launch_after reports it there, and the
// kernels after it would run on what an earlier call left in the workspace.
// Zero `bytes` (rounded up to 16) at the 16-byte aligned p.
[[nodiscard]] cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t st);
// The largest |x| (IEEE bits) of every row of A (M vectors) and column of B
// (N), in one launch; a null maxA or maxB leaves that operand out.  zeroed:
// the outputs are zero already.
template <typename T>
[[nodiscard]] cudaError_t launch_scan(const T* A, int64_t ldA, bool a_kcontig, int64_t M, unsigned long long* maxA, const T* B,
                 int64_t ldB, bool b_kcontig, int64_t N, unsigned long long* maxB, int64_t k, int cw, bool zeroed,
                 int* status, cudaStream_t st);
// One operand, zeroed here.
template <typename T>
[[nodiscard]] inline cudaError_t launch_scan_one(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k, int cw,
                            unsigned long long* maxbits, int* status, cudaStream_t st) {
  return launch_scan<T>(X, ld, kcontig, rows, maxbits, static_cast<const T*>(nullptr), 1, false, 0, nullptr, k, cw,
                        false, status, st);
}
template <typename T>
[[nodiscard]] cudaError_t launch_split_I(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k, int p,
                    const unsigned long long* maxbits, int8_t* hat, int32_t* E, cudaStream_t st,
                    bool f8 = false);
template <typename T>
[[nodiscard]] cudaError_t launch_split_II(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k, int nm, int b,
                     int cw, const ModTables& tabs, const unsigned long long* maxbits, int8_t* res,
                     int32_t* E, cudaStream_t st, const unsigned long long* acc = nullptr, bool bf16 = false);
// Norm-based Scheme II scaling: the sums of squares of both operands' vectors
// in one launch, exact in any order (maxima from launch_scan; acc: two words
// per vector, zeroed; null: that operand is left out).
template <typename T>
[[nodiscard]] cudaError_t launch_norm(const T* A, int64_t ldA, bool a_kcontig, int64_t M, const unsigned long long* maxA,
                 unsigned long long* accA, const T* B, int64_t ldB, bool b_kcontig, int64_t N,
                 const unsigned long long* maxB, unsigned long long* accB, int64_t k, int cw, cudaStream_t st);
void host_norm_halves_II(int nm, int* hA, int* hB);

// Output modes of the Scheme I kernel.
enum GemmOut : int { OUT_F64 = 0, OUT_F32 = 1, OUT_PARTIALS = 2 };

struct GemmIArgs {
  const CUtensorMap* descA;  // host copies, passed to the kernel by value
  const CUtensorMap* descB;
  int M, N;
  int nk32;     // number of 32-wide K-chunks
  int kc32;     // fold interval in K-chunks (K_c / 32)
  const int32_t* EA;
  const int32_t* FB;
  double alpha, beta;
  void* C;
  int64_t ldc;
  int32_t* partials;
  int* status;
  int num_sms;
};
cudaError_t launch_gemm_I(int p, int out_mode, const GemmIArgs& a, cudaStream_t st, bool f8 = false);
// Scheme I on E4M3 slices with tcgen05 / TMEM (128 x 32 output tiles).
cudaError_t launch_gemm_f8tc(int p, int out_mode, const GemmIArgs& a, cudaStream_t st);

// Scheme I on the bf16 tensor cores (tri_core.cuh): layout of one product,
// the split of one operand, and the GEMM (part 1) and combine (part 2)
// kernels.
struct TriLayout {
  int64_t tiles_m, tiles_n, kpad;
  int64_t nkc, kcs;   // K ranges of the int32 sums, 64-deep chunks per range
  int64_t planes;     // int32 output planes
  bool one;           // one plane pair per output plane, else one group of them
  size_t Cs_bytes;
};
// one: 1 or 0 fixes `one`, -1 leaves it to the product's size.
TriLayout tri_layout(int64_t M, int64_t N, int64_t k, int p, int one = -1);
// The products of the recentring constants alone (part of every S), 128 bits.
void tri_const(int p, int64_t K, uint64_t* lo, uint64_t* hi);
int tri_tile_m();
int tri_tile_n();
int tri_num_planes(int p);
int tri_num_units(int p);  // int32 output planes with one unit per group
struct GemmTriArgs {
  TriLayout L;
  const CUtensorMap* descA;
  const CUtensorMap* descB;
  int box_bytes;  // of one 64-deep chunk: the rows of both maps' boxes x 128 bytes
  int M, N;
  int64_t K;
  int32_t* Cs;
  const int32_t* sumA;
  const int32_t* sumB;
  const int32_t* EA;
  const int32_t* FB;
  double alpha, beta;
  void* C;
  int64_t ldc;
  int* status;
  int num_sms;
};
cudaError_t launch_gemm_I_tc(int p, int out_mode, const GemmTriArgs& a, cudaStream_t st, int part);
template <typename T>
[[nodiscard]] cudaError_t launch_split_tri(const T* X, int64_t ld, bool kcontig, int64_t rows, int64_t k, int p,
                      const unsigned long long* maxbits, uint16_t* planes, int32_t* E, int32_t* sums, int num_sms,
                      cudaStream_t st);

// Scheme II kernel modes.
enum GemmIIOut : int { II_F64 = 0, II_F32 = 1, II_RESIDUES = 2, II_Z3M = 3, II_C3M = 4 };

struct GemmIIArgs {
  const CUtensorMap* descA;
  const CUtensorMap* descB;
  int M, N, K;
  int nk32;
  int rowsA_pad, rowsB_pad;  // plane heights in the stacked residue matrices
  int nm;
  int escale;                 // -2b
  const int32_t* EA;
  const int32_t* FB;
  double alpha_re, alpha_im, beta_re, beta_im;
  void* C;
  int64_t ldc;
  uint8_t* residues;
  int* status;
  int num_sms;
  int cluster;       // tcgen05 kernel: CTAs per GEMM tile (2: a CTA pair, cta_group::2; 1: one CTA)
  uint8_t* scratch;  // tcgen05 kernel: the residue planes
};
cudaError_t launch_gemm_II(int out_mode, const GemmIIArgs& a, const ModTables& mt,
                           const CrtTables& ct, cudaStream_t st);
// Scheme II on bf16 residue planes with tcgen05 / TMEM (256 x 256 tiles on
// CTA pairs, or 128 x 256 on single CTAs; modulus-major), then the CRT
// kernel; modes II_F64, II_F32, II_Z3M, II_C3M.  GemmIIArgs::scratch: gemm_II_tc_residue_bytes(M, N, nm, complex,
// cluster) bytes of device memory for the residue planes.  part: 1 launches
// the residue GEMM, 2 the CRT kernel (after the residue GEMM on the same
// stream), 3 both.
cudaError_t launch_gemm_II_tc(int out_mode, const GemmIIArgs& a, const ModTables& mt,
                              const CrtPairTables& ct, cudaStream_t st, int part = 3);
int gemm_II_tc_tile_m();
int gemm_II_tc_tile_n();
size_t gemm_II_tc_residue_bytes(int64_t M, int64_t N, int nm, bool is_complex, int cluster);
int gemm_II_tc_cluster(int64_t M, int64_t K);

// Tensor map for a row-major byte matrix [rows][cols] read in boxes of
// box_bytes x box_rows: 32-byte boxes with 32-byte swizzling, or 128-byte
// boxes with 128-byte swizzling.
bool make_tmap_i8(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows,
                  uint32_t box_rows, uint32_t box_bytes = 32);

}  // namespace emu
