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
#include "tri_kernels.cuh"

namespace emu {
namespace {

struct KParamsTri {
  CUtensorMap tA;  // planes as bytes: 128-byte x 128-row boxes (fewer if M is less), 128-byte swizzle
  CUtensorMap tB;  // 128-byte x 256-row boxes (fewer if N is less)
  TriPlan tp;
  int nst, kcs, nkc;  // 64-deep chunks of a plane; chunks per K range; K ranges
  int tiles_m, tiles_n;  // 128-row and 256-column tiles
  int M, N;  // rows of A's planes and of B's
  int box_bytes;
  int32_t* Cs;  // output planes, tile by tile (tri_elem)
  int* status;
};

// Work items (unit, K range, tile) in that order; a unit's plane pairs.
struct TriWork {
  const KParamsTri& kp;
  __device__ __forceinline__ bool at(int r, int cid, int ncl, bf16g::Item& t) const {
    const int tiles = kp.tiles_m * kp.tiles_n, per = kp.nkc * tiles;
    int i = bf16g::item_index(r, cid, ncl);
    if (i >= kp.tp.nunits * per) return false;
    t.unit = i / per;
    i -= t.unit * per;
    t.aux = i / tiles;  // K range
    tile_coords16(i - t.aux * tiles, kp.tiles_m, kp.tiles_n, t.tm, t.tn);
    const TriUnit u = kp.tp.unit[t.unit];
    t.np = u.count;
    t.seg = u.sums ? bf16g::Cfg<false>::kSeg16 : bf16g::Cfg<false>::kSeg14;
    t.k0 = t.aux * kp.kcs;
    t.k1 = t.k0 + kp.kcs < kp.nst ? t.k0 + kp.kcs : kp.nst;
    t.cols = bf16g::tile_cols(kp.N, t.tn);
    return true;
  }
  __device__ __forceinline__ int ya(const bf16g::Item& t, int q) const {
    return kp.tp.pa[kp.tp.unit[t.unit].first + q] * kp.M + t.tm * kBM;
  }
  __device__ __forceinline__ int yb(const bf16g::Item& t, int q) const {
    return kp.tp.pb[kp.tp.unit[t.unit].first + q] * kp.N + t.tn * kBN;
  }
  __device__ __forceinline__ const CUtensorMap* tA(const bf16g::Item&) const { return &kp.tA; }
  __device__ __forceinline__ const CUtensorMap* tB(const bf16g::Item&) const { return &kp.tB; }
  __device__ __forceinline__ int bytes(const bf16g::Item&) const { return kp.box_bytes; }
  // where this item's sums go
  __device__ __forceinline__ int32_t* tile_of(const bf16g::Item& t) const {
    const int64_t plane = static_cast<int64_t>(kp.tp.unit[t.unit].out) * kp.nkc + t.aux;
    return kp.Cs + (plane * kp.tiles_m * kp.tiles_n + static_cast<int64_t>(t.tn) * kp.tiles_m + t.tm) * kTileElems;
  }
  __device__ __forceinline__ int rows(const bf16g::Item&) const { return kp.M; }
};

__global__ void __launch_bounds__(bf16g::kThreads, 1) gemm_I_tc_kernel(const __grid_constant__ KParamsTri kp) {
  tri_gemm(TriWork{kp}, kp.status);
}

// ---------------------------------------------------------------- combine
// A block combines a 32 x 32 patch (combine_patch).
template <int P, bool ONE>
__global__ void __launch_bounds__(256) combine_I_kernel(const __grid_constant__ KParamsTriComb kp) {
  grid_begin();
  combine_patch<P, ONE>(kp, static_cast<int>(blockIdx.x));
}

// ---------------------------------------------------------------- plan
template <int P>
cudaError_t launch_combine(const KParamsTriComb& kp, bool one, cudaStream_t st) {
  const unsigned grid = static_cast<unsigned>(kp.tiles_m * kp.tiles_n * kp.pr * kp.pc);
  return one ? launch_after(combine_I_kernel<P, true>, grid, 256, st, kp)
             : launch_after(combine_I_kernel<P, false>, grid, 256, st, kp);
}

}  // namespace

int tri_tile_m() { return kBM; }
int tri_tile_n() { return kBN; }
int tri_num_planes(int p) {
  constexpr PlaneCounts counts{};
  return counts.n[p];
}

int tri_num_units(int p) { return plan_of(p, false).nunits; }

void tri_const(int p, int64_t K, uint64_t* lo, uint64_t* hi) {
  // 2^14 K sum_{i,j>=1, i+j<p} 256^(p-1-i-j): s - 1 pairs with i + j = s
  unsigned __int128 w = 0;
  for (int s = 0; s < p; ++s) w = w * 256 + static_cast<unsigned>(s > 1 ? s - 1 : 0);
  w = w * static_cast<unsigned __int128>(K) << 14;
  *lo = static_cast<uint64_t>(w);
  *hi = static_cast<uint64_t>(w >> 64);
}

TriLayout tri_layout(int64_t M, int64_t N, int64_t k, int p, int one) {
  TriLayout L{};
  L.tiles_m = (M + kBM - 1) / kBM;
  L.tiles_n = (N + kBN - 1) / kBN;
  L.kpad = (k + 63) / 64 * 64;
  const int64_t nst = L.kpad / 64;
  // One unit per s and kind (fewest planes) when its items fill the GPU
  // several times; one unit per plane pair for smaller products, whose time
  // is the longest item's.
  L.one = one >= 0 ? one != 0 : L.tiles_m * L.tiles_n * plan_of(p, false).nunits < 4 * kSms;
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
    kp.box_bytes = a.box_bytes;
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
  kc.pr = patch_rows(a.M);
  kc.pc = patch_cols(a.N);
  kc.sumA = a.sumA;
  kc.sumB = a.sumB;
  tri_const(p, a.K, &kc.const_lo, &kc.const_hi);
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
