// bf16_gemm.cuh -- the persistent tcgen05 kind::f16 main loop shared by the
// Scheme II residue GEMM and the Scheme I digit triangle: exact integer
// products of bf16 planes, FP32 accumulators in tensor memory that are
// drained before a sum could leave the exact range.
//
// Two forms.  PAIR: a 256 x 256 tile on a pair of CTAs (a cluster of two on
// neighbouring SMs, tcgen05.mma.cta_group::2): one 256 x 256 x 16 MMA per
// K-step, issued by the even CTA, reads the 128 rows of A that each CTA holds
// and the 256 columns of B of which each CTA holds half, and leaves rows
// 0-127 of the product in the even CTA's TMEM and rows 128-255 in the odd
// one's.  Single: a 128 x 256 tile on one CTA.
//
// What bounds them: shared-memory bandwidth, 128 B per clock and SM.  Per
// K-step of 16 (128 clocks of tensor work) an SM of the single form receives
// 12 KB by TMA and reads 12 KB, 1.5 times what 128 clocks deliver; the pair
// form moves 8 + 8 KB, which just fits.  Main loop alone, all SMs, operands
// from L2 and HBM: single 858 clocks per 64-deep stage (1.40 PFLOP/s), pair
// 597 (1.92 PFLOP/s), ideal 512.  The pair form needs stages 128 deep (three
// of 64 KB): with 64-deep stages the issuing thread meets a barrier every
// 512 clocks, whose round trip over both CTAs drains the MMA queue (888
// clocks); the single form does not gain from deeper stages (898).
// While the MMAs of the pair form run, tensor-memory reads wait for gaps
// between them: a drain takes about 3500 clocks instead of 1800, so the pair
// form pays only where segments are long (digits and residues, 7168 clocks),
// not for digit sums (2048).
//
// Roles (320 threads per CTA): warps 0-7 drain (warp w: TMEM lanes = tile
// rows 32 (w % 4) .., columns 128 (w / 4) ..), warp 8 lane 0 TMA, warp 9 TMEM
// allocation and (lane 0 of the even CTA) MMAs.  Sixteen drain warps of 64
// columns were 3-6 % slower in both forms.  Two FP32 accumulators take
// all 512 TMEM columns of each CTA and alternate between segments, so the
// MMAs of one segment overlap the drain of the last.  All waits are bounded;
// a timeout sets the status word, raises the abort flag of both CTAs of a
// pair for the other roles, and the TMEM is still released.
//
// Work: a policy W with
//   bool at(r, cid, ncl, item): the r-th item of CTA (pair) cid of ncl; false
//     after the last one.  An item: plane-pair count `np`, K range [k0, k1) in
//     64-deep chunks, first 128-row tile tm (of the even CTA), column tile tn,
//     segment length `seg` in stages, columns `cols` that the MMAs compute
//   int ya(item, q), yb(item, q): first row of A's tile (the even CTA's) and
//     of B's tile in the stacked planes, for plane pair q
//   const CUtensorMap* tA(item), tB(item); int bytes(item): of one chunk's boxes
#pragma once
#include "emu_internal.h"
#include "tc_core.cuh"

namespace emu {
namespace bf16g {

constexpr int kBM = 128, kBN = 256;  // accumulator tile of one CTA: TMEM lanes x FP32 columns
constexpr int kDrainWarps = 8;
constexpr int kDrainCols = kBN / (kDrainWarps / 4);  // columns of one drain warp
constexpr int kProducerWarp = kDrainWarps, kMmaWarp = kDrainWarps + 1;
constexpr int kThreads = 32 * (kDrainWarps + 2);

template <bool PAIR>
struct Cfg {
  static constexpr int kKS = PAIR ? 2 : 1;                // 64-deep chunks per stage
  static constexpr int kRowsB = PAIR ? kBN / 2 : kBN;     // B rows (output columns) this CTA loads
  static constexpr int kBlkA = kBM * 128;                 // one chunk: 128 rows x 64 bf16, 128-byte rows
  static constexpr int kBlkB = kRowsB * 128;
  static constexpr int kChunkBytes = kBlkA + kBlkB;
  static constexpr int kStageBytes = kKS * kChunkBytes;
  static constexpr int kStages = PAIR ? 3 : 4;
  static constexpr int kSmem = kStages * kStageBytes + 1024 + 256;
  // stages per exact FP32 segment: sums of 2^14 (digits, residues; at most
  // 960 of them) and of 2^16 (digit sums; 256)
  static constexpr int kSeg14 = PAIR ? 7 : 15, kSeg16 = PAIR ? 2 : 4;
  static_assert(kSmem <= 232448, "shared memory");
  static_assert(kChunkBytes % 1024 == 0, "chunks keep the 1024-byte swizzle alignment");
  static_assert(kSeg14 * kKS * 64 * 16384 < (1 << 24) && kSeg16 * kKS * 64 * 65536 <= (1 << 24),
                "segment sums must stay exact in FP32");
};

struct Item {
  int unit, np, k0, k1, seg, tm, tn, cols, aux, prob;
};

// Stages of one item: every plane pair has its own, the last of each may
// hold fewer than kKS chunks.
template <bool PAIR>
__device__ __forceinline__ int stages_of(const Item& t) {
  return t.np * ((t.k1 - t.k0 + Cfg<PAIR>::kKS - 1) / Cfg<PAIR>::kKS);
}

// Index of CTA (pair) cid's item in round r: odd rounds run backwards, which
// evens out the sums when the items are sorted by length.
__device__ __forceinline__ int item_index(int r, int cid, int ncl) {
  return r * ncl + ((r & 1) ? ncl - 1 - cid : cid);
}

struct Ctx {
  uint8_t* smem;
  uint32_t base;
  uint64_t *full, *empty, *acc_full, *acc_empty;
  uint32_t tmem;
  uint32_t crank;
  int cid, ncl, warp, lane;
  AbortFlag ab;
};

template <bool PAIR>
__device__ __forceinline__ Ctx setup(uint8_t* smem_raw) {
  using C = Cfg<PAIR>;
  Ctx c;
  const uint32_t raw = smem_u32(smem_raw);
  c.base = (raw + 1023u) & ~1023u;
  c.smem = smem_raw + (c.base - raw);
  c.full = reinterpret_cast<uint64_t*>(c.smem + C::kStages * C::kStageBytes);
  c.empty = c.full + C::kStages;
  c.acc_full = c.empty + C::kStages;  // two accumulators
  c.acc_empty = c.acc_full + 2;
  uint32_t* slot = reinterpret_cast<uint32_t*>(c.acc_empty + 2);
  volatile int* abort_local = reinterpret_cast<volatile int*>(slot + 1);
  c.warp = threadIdx.x >> 5;
  c.lane = threadIdx.x & 31;
  c.crank = PAIR ? cluster_ctarank() : 0u;  // 0: the pair's MMA-issuing CTA
  c.cid = PAIR ? static_cast<int>(cluster_id_x()) : static_cast<int>(blockIdx.x);
  c.ncl = PAIR ? static_cast<int>(cluster_count_x()) : static_cast<int>(gridDim.x);
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(&c.full[s], 1);   // the even CTA's expect-tx arrival (+ the bytes of both CTAs)
      mbar_init(&c.empty[s], 1);  // one MMA commit
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&c.acc_full[b], 1);
      mbar_init(&c.acc_empty[b], PAIR ? 2 * kDrainWarps : kDrainWarps);  // one arrival per drain warp
    }
    *abort_local = 0;
    fence_mbar_init();
  }
  if (c.warp == kMmaWarp) {  // the whole warp allocates the tensor memory (both CTAs of a pair)
    tmem_alloc_all<PAIR>(slot);
    tc_fence_before();
  }
  // barriers and flags initialised in both CTAs before either touches the peer's
  if (PAIR)
    cluster_sync_all();
  else
    __syncthreads();
  tc_fence_after();
  grid_begin();  // barriers and tensor memory were set up while the kernel before ended
  c.tmem = *slot;
  c.ab.local = abort_local;
  c.ab.peer = PAIR ? cluster_addr(smem_u32(const_cast<int*>(abort_local)), c.crank ^ 1u) : 0u;
  return c;
}

// Signal `bar` (of both CTAs of a pair) once every MMA issued so far has completed.
template <bool PAIR>
__device__ __forceinline__ void commit(uint64_t* bar) {
  if constexpr (PAIR)
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"(static_cast<uint16_t>(3))
        : "memory");
  else
    umma_commit(bar);
}

// The producer thread (one of each CTA).
template <bool PAIR, class W>
__device__ __forceinline__ void produce(const Ctx& c, const W& w, int* status) {
  using C = Cfg<PAIR>;
  uint32_t j = 0;
  bool stop = false;
  Item t;
  for (int r = 0; !stop && w.at(r, c.cid, c.ncl, t); ++r) {
    const CUtensorMap *const tA = w.tA(t), *const tB = w.tB(t);
    tma_prefetch_desc(tA);
    tma_prefetch_desc(tB);
    const int bytes = (PAIR ? 2 : 1) * w.bytes(t);
    // each CTA of a pair holds half of the columns the MMAs read
    const int half = PAIR ? static_cast<int>(c.crank) * (t.cols / 2) : 0;
    for (int q = 0; q < t.np && !stop; ++q) {
      const int ya = w.ya(t, q) + static_cast<int>(c.crank) * kBM, yb = w.yb(t, q) + half;
      for (int ks = t.k0; ks < t.k1; ks += C::kKS, ++j) {
        const uint32_t stage = j % C::kStages;
        if (j >= static_cast<uint32_t>(C::kStages) &&
            !wait_pair(&c.empty[stage], ((j / C::kStages) & 1u) ^ 1u, c.ab, status)) {
          stop = true;
          break;
        }
        uint8_t* s = c.smem + stage * C::kStageBytes;
        const int parts = t.k1 - ks < C::kKS ? t.k1 - ks : C::kKS;
        if (c.crank == 0) mbar_arrive_expect_tx(&c.full[stage], parts * bytes);
        // both CTAs' bytes are counted on the even CTA's barrier
        const uint32_t bar = PAIR ? cluster_addr(smem_u32(&c.full[stage]), 0u) : 0u;
#pragma unroll
        for (int k = 0; k < C::kKS; ++k) {
          if (k >= parts) break;
          uint8_t* const sA = s + k * C::kBlkA;
          uint8_t* const sB = s + C::kKS * C::kBlkA + k * C::kBlkB;
          if (PAIR) {
            tma_load_2d_pair(sA, tA, bar, (ks + k) * 128, ya);
            tma_load_2d_pair(sB, tB, bar, (ks + k) * 128, yb);
          } else {
            tma_load_2d(sA, tA, &c.full[stage], (ks + k) * 128, ya);
            tma_load_2d(sB, tB, &c.full[stage], (ks + k) * 128, yb);
          }
        }
      }
    }
  }
  // Drain: wait until the last MMA commits have arrived on this CTA's stage
  // barriers (a pair's odd CTA gets them from the even one), so that none
  // lands after the CTA exits.
  if (!stop && PAIR) {
    for (uint32_t jj = j; jj < j + C::kStages; ++jj) {
      if (jj < static_cast<uint32_t>(C::kStages)) continue;
      const uint32_t stage = jj % C::kStages;
      if (!wait_pair(&c.empty[stage], ((jj / C::kStages) & 1u) ^ 1u, c.ab, status)) break;
    }
  }
}

// The MMA thread (of the even CTA).
template <bool PAIR, class W>
__device__ __forceinline__ void issue(const Ctx& c, const W& w, int* status) {
  using C = Cfg<PAIR>;
  uint32_t it = 0, seg = 0;
  bool stop = false;
  bool ready = false;  // the probe after the previous stage's MMAs already saw this stage's data
  Item t;
  for (int r = 0; !stop && w.at(r, c.cid, c.ncl, t); ++r) {
    const uint32_t idesc = idesc_bf16(PAIR ? 2 * kBM : kBM, t.cols);
    const int per = (t.k1 - t.k0 + C::kKS - 1) / C::kKS, n = t.np * per;
    const int last_parts = t.k1 - t.k0 - (per - 1) * C::kKS;  // chunks of a plane pair's last stage
    int left = 0, ks = 0;  // stages left in this segment; stage within the plane pair
    for (int x = 0; x < n; ++x, ++it) {
      const bool first = left == 0;
      const uint32_t b = seg & 1u;
      if (first) {
        left = t.seg < n - x ? t.seg : n - x;
        if (seg >= 2) {  // the drain warps must have read this accumulator's last segment
          if (!wait_pair(&c.acc_empty[b], ((seg >> 1) - 1) & 1u, c.ab, status, PAIR)) {
            stop = true;
            break;
          }
          tc_fence_after();
        }
      }
      const uint32_t stage = it % C::kStages;
      if (!ready && !wait_pair(&c.full[stage], (it / C::kStages) & 1u, c.ab, status)) {
        stop = true;
        break;
      }
      tc_fence_after();
      const uint32_t s = c.base + stage * C::kStageBytes;
      const int parts = ++ks == per ? last_parts : C::kKS;
      if (ks == per) ks = 0;
#pragma unroll
      for (int k = 0; k < C::kKS; ++k) {
        if (k >= parts) break;
        const uint32_t sA = s + k * C::kBlkA, sB = s + C::kKS * C::kBlkA + k * C::kBlkB;
#pragma unroll
        for (int q = 0; q < 4; ++q)  // four K-steps of 16 inside the 128-byte rows
          umma_bf16<PAIR>(c.tmem + b * kBN, smem_desc_k128(sA + 32 * q), smem_desc_k128(sB + 32 * q), idesc,
                          (first && k == 0 && q == 0) ? 0u : 1u);
      }
      // Probe (without blocking) the next stage while these MMAs are queued,
      // so that its MMAs follow at once when the data is there.  After the
      // CTA's last stage the probe reads an older phase; its answer is not
      // used.
      ready = mbar_test_wait(&c.full[(it + 1) % C::kStages], ((it + 1) / C::kStages) & 1u);
      commit<PAIR>(&c.empty[stage]);
      if (--left == 0) {
        commit<PAIR>(&c.acc_full[b]);
        ++seg;
      }
    }
  }
}

// Wait (one lane polls, the warp follows) for segment `seg`'s accumulator.
__device__ __forceinline__ bool wait_segment(const Ctx& c, uint32_t seg, int* status) {
  bool ok = true;
  if (c.lane == 0) ok = wait_pair(&c.acc_full[seg & 1u], (seg >> 1) & 1u, c.ab, status);
  ok = __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0;
  __syncwarp();
  if (ok) tc_fence_after();
  return ok;
}

// This warp has read accumulator seg & 1: the MMAs may refill it.
template <bool PAIR>
__device__ __forceinline__ void release_segment(const Ctx& c, uint32_t seg) {
  tc_fence_before();
  __syncwarp();
  if (c.lane == 0) {
    if (PAIR)
      mbar_arrive_cluster(cluster_addr(smem_u32(&c.acc_empty[seg & 1u]), 0u));
    else
      mbar_arrive(&c.acc_empty[seg & 1u]);
  }
}

// TMEM address of this drain warp's first column of accumulator 0.
__device__ __forceinline__ uint32_t drain_addr(const Ctx& c) {
  return c.tmem + (static_cast<uint32_t>((c.warp & 3) * 32) << 16) + static_cast<uint32_t>((c.warp >> 2) * kDrainCols);
}

template <bool PAIR>
__device__ __forceinline__ void finish(const Ctx& c) {
  tc_fence_before();
  // no CTA of a pair leaves while the other may still touch its shared or tensor memory
  if (PAIR)
    cluster_sync_all();
  else
    __syncthreads();
  if (c.warp == kMmaWarp) {
    tc_fence_after();
    tmem_free_all<PAIR>(c.tmem);
  }
}

// Columns of column tile tn that the MMAs compute: of the last tile only as
// many as n needs, in steps of 32.
__device__ __forceinline__ int tile_cols(int n, int tn) {
  const int left = n - tn * kBN;
  return left >= kBN ? kBN : (left + 31) & ~31;
}

// Launch `kernel` on nitems items: one CTA (pair) per SM (two SMs).
template <bool PAIR, class K, class... Args>
cudaError_t launch(K kernel, int64_t nitems, int num_sms, cudaStream_t st, const Args&... args) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<PAIR>::kSmem);
  if (e != cudaSuccess) return e;
  const int64_t most = PAIR ? num_sms / 2 : num_sms;
  const int64_t n = nitems < most ? nitems : most;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 2;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(PAIR ? 2 * n : n));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = Cfg<PAIR>::kSmem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = PAIR ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace bf16g
}  // namespace emu
