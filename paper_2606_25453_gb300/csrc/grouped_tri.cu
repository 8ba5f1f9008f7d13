// grouped_tri.cu -- many independent Scheme I products as bf16 digit triangles
// (tri_core.cuh): one split, one persistent GEMM and one combine launch for
// the whole batch.
//
// The GEMM's work list holds every product's (unit, K range, tile) items,
// longest first; CTA c takes items c, 2 G - 1 - c, 2 G + c, .. of the G CTAs,
// which evens out the sums without a queue.  A product narrower than a tile
// loads only the rows it has (its tensor maps' boxes) and computes only its
// columns in steps of 32.  On 512 products (M, N in [32, 1024], K in [64,
// 2048], p = 6) this replaces the mma.sync launches, whose 155 TOP/s bounded
// the batch at 8 ms of 9.5.
#include <algorithm>

#include "grouped_tri.h"
#include "split_tri_core.cuh"
#include "tri_kernels.cuh"

namespace emu {

struct GTriProb {
  const double *A, *B;
  double* C;
  int64_t lda, ldb, ldc, kpad;
  double alpha, beta;
  unsigned long long *maxA, *maxB;
  int32_t *EA, *FB, *sumA, *sumB;
  uint16_t *planesA, *planesB;
  int32_t* Cs;
  uint64_t const_lo, const_hi;
  int M, N, K, nst, kcs, nkc, tiles_m, tiles_n, box_bytes;
};

namespace {

constexpr int kSplitRun = 8;  // groups of 128 elements along K per split block

// Blocks [0, startA[count]): eight rows of A x kSplitRun groups of 128
// elements, one row per warp; the rest: 32 columns of B x as many through
// shared memory.  HBM bound in principle (2 bytes per plane written); what
// costs is each block's chain of dependent loads (product, table entry,
// exponent, elements), hence several groups per block: the batch above took
// 4.59 ms with one group per block and a binary search for the product, 4.01
// with this and the search by whole warps.  Blocks per SM: what the compiler
// reaches by itself, and at p = 6 three instead of two (80 registers for 97; that
// batch 3.95 ms against 4.26).
template <int P>
__global__ void __launch_bounds__(256, P <= 4 ? 4 : P <= 6 ? 3 : 2) grouped_split_tri_kernel(const GTriProb* __restrict__ probs, int count,
                                                                   const int* __restrict__ startA,
                                                                   const int* __restrict__ startB) {
  __shared__ uint64_t tile[32][133];
  __shared__ int ssum[32][P], sE[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int blk = blockIdx.x;
  const int totA = startA[count];
  const bool first = blk < totA;
  if (!first) blk -= totA;
  const int* const start = first ? startA : startB;
  const int pi = find_prob(start, count, blk);
  const GTriProb& pr = probs[pi];
  const int64_t rows = first ? pr.M : pr.N, kpad = pr.kpad, K = pr.K;
  const int nrun = (static_cast<int>((kpad + 127) / 128) + kSplitRun - 1) / kSplitRun;
  const int local = blk - start[pi];
  const int64_t r0 = static_cast<int64_t>(local / nrun) * (first ? 8 : 32), hb = (local % nrun) * (kSplitRun * 128);
  const int64_t hend = min(hb + kSplitRun * 128, kpad);
  const int64_t plane = rows * kpad;
  if (first) {
    const int64_t r = r0 + warp;
    if (r >= rows) return;
    const double* const X = pr.A + r * pr.lda;
    const bool vec = vec16_ok(pr.A, pr.lda);
    uint16_t* const dst = pr.planesA + r * kpad;
    const int E = exp_from_maxbits(pr.maxA, r, rows);
    if (hb == 0 && lane == 0) pr.EA[r] = E;
    int sum[P];
#pragma unroll
    for (int t = 0; t < P; ++t) sum[t] = 0;
    for (int64_t h0 = hb + lane * 4; h0 < hend; h0 += 128) {
      uint64_t bits[4];
      load4_kcontig(X, h0, K, true, vec, bits);
      digits4<P>(bits, E, live_count(h0, K), dst + h0, plane, sum);
    }
    __syncwarp();
    int mine = 0;
#pragma unroll
    for (int t = 0; t < P; ++t) {
      const int s = __reduce_add_sync(0xFFFFFFFFu, sum[t]);
      if (lane == t) mine = s;
    }
    if (lane < P) atomicAdd(pr.sumA + lane * rows + r, mine);
    return;
  }
  const bool vec = vec16_ok(pr.B, pr.ldb);
  const double* const X = pr.B;
  const int64_t ld = pr.ldb;
  for (int i = threadIdx.x; i < 32 * P; i += 256) (&ssum[0][0])[i] = 0;
  if (threadIdx.x < 32 && r0 + threadIdx.x < rows) {
    const int E = exp_from_maxbits(pr.maxB, r0 + threadIdx.x, rows);
    sE[threadIdx.x] = E;
    if (hb == 0) pr.FB[r0 + threadIdx.x] = E;
  }
  for (int64_t hbase = hb; hbase < hend; hbase += 128) {
    __syncthreads();  // the previous group is done with the tile
    fill_tile_strided(tile, X, ld, rows, K, r0, hbase, vec);
    __syncthreads();
    const int64_t h0 = hbase + lane * 4;
#pragma unroll 1
    for (int rl = warp; rl < 32; rl += 8) {
      const int64_t r = r0 + rl;
      if (r >= rows) break;
      int sum[P];
#pragma unroll
      for (int t = 0; t < P; ++t) sum[t] = 0;
      if (h0 < kpad) {
        uint64_t bits[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) bits[q] = tile[rl][q * 33 + lane];
        digits4<P>(bits, sE[rl], live_count(h0, K), pr.planesB + r * kpad + h0, plane, sum);
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
  for (int i = threadIdx.x; i < 32 * P; i += 256) {
    const int rl = i % 32, t = i / 32;
    if (r0 + rl < rows) atomicAdd(pr.sumB + t * rows + r0 + rl, ssum[rl][t]);
  }
}

struct KParamsGTri {
  TriPlan tp;
  const GTriProb* probs;
  const CUtensorMap* maps;
  const int4* items;  // {product, unit | K range << 8, row tile, column tile}
  int nitems;
  int* status;
};

struct GTriWork {
  const KParamsGTri& kp;
  __device__ __forceinline__ bool at(int r, int cid, int ncl, bf16g::Item& t) const {
    const int i = bf16g::item_index(r, cid, ncl);
    if (i >= kp.nitems) return false;
    const int4 e = __ldg(kp.items + i);
    const GTriProb& pr = kp.probs[e.x];
    t.prob = e.x;
    t.unit = e.y & 0xFF;
    t.aux = e.y >> 8;
    t.tm = e.z;
    t.tn = e.w;
    const TriUnit u = kp.tp.unit[t.unit];
    t.np = u.count;
    t.seg = u.sums ? bf16g::Cfg<false>::kSeg16 : bf16g::Cfg<false>::kSeg14;
    t.k0 = t.aux * pr.kcs;
    t.k1 = t.k0 + pr.kcs < pr.nst ? t.k0 + pr.kcs : pr.nst;
    t.cols = bf16g::tile_cols(pr.N, t.tn);
    return true;
  }
  __device__ __forceinline__ int ya(const bf16g::Item& t, int q) const {
    return kp.tp.pa[kp.tp.unit[t.unit].first + q] * kp.probs[t.prob].M + t.tm * kBM;
  }
  __device__ __forceinline__ int yb(const bf16g::Item& t, int q) const {
    return kp.tp.pb[kp.tp.unit[t.unit].first + q] * kp.probs[t.prob].N + t.tn * kBN;
  }
  __device__ __forceinline__ const CUtensorMap* tA(const bf16g::Item& t) const { return kp.maps + 2 * t.prob; }
  __device__ __forceinline__ const CUtensorMap* tB(const bf16g::Item& t) const { return kp.maps + 2 * t.prob + 1; }
  __device__ __forceinline__ int bytes(const bf16g::Item& t) const { return kp.probs[t.prob].box_bytes; }
  __device__ __forceinline__ int32_t* tile_of(const bf16g::Item& t) const {
    const GTriProb& pr = kp.probs[t.prob];
    const int64_t plane = static_cast<int64_t>(kp.tp.unit[t.unit].out) * pr.nkc + t.aux;
    return pr.Cs + (plane * pr.tiles_m * pr.tiles_n + static_cast<int64_t>(t.tn) * pr.tiles_m + t.tm) * kTileElems;
  }
  __device__ __forceinline__ int rows(const bf16g::Item& t) const { return kp.probs[t.prob].M; }
};

__global__ void __launch_bounds__(bf16g::kThreads, 1) gemm_I_grouped_tc_kernel(const __grid_constant__ KParamsGTri kp) {
  tri_gemm(GTriWork{kp}, kp.status);
}

// Two blocks per SM at p = 8 with one plane per group, where the compiler would
// take 152 registers for one (512 products, M, N <= 1024, K <= 2048: 5.63 ms
// against 6.19); below it reaches two by itself, and with one plane per pair
// (small batches) 128 registers spill.
template <int P, bool ONE>
__global__ void __launch_bounds__(256, P == 8 && !ONE ? 2 : 0) grouped_combine_kernel(const GTriProb* __restrict__ probs, int count,
                                                              const int* __restrict__ startC) {
  const int pi = find_prob(startC, count, blockIdx.x);
  const GTriProb& pr = probs[pi];
  KParamsTriComb kp;
  kp.Cs = pr.Cs;
  kp.nkc = pr.nkc;
  kp.tiles_m = pr.tiles_m;
  kp.tiles_n = pr.tiles_n;
  kp.M = pr.M;
  kp.N = pr.N;
  kp.pr = patch_rows(pr.M);
  kp.pc = patch_cols(pr.N);
  kp.sumA = pr.sumA;
  kp.sumB = pr.sumB;
  kp.const_lo = pr.const_lo;
  kp.const_hi = pr.const_hi;
  kp.EA = pr.EA;
  kp.FB = pr.FB;
  kp.escale = -14 - 8 * (P - 1);
  kp.alpha = pr.alpha;
  kp.beta = pr.beta;
  kp.C = pr.C;
  kp.ldc = pr.ldc;
  kp.plain = pr.alpha == 1.0 && pr.beta == 0.0;
  kp.f32 = 0;
  combine_patch<P, ONE>(kp, static_cast<int>(blockIdx.x) - startC[pi]);
}

size_t al256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

// One product's share of the workspace.
struct Share {
  TriLayout L;
  size_t zero, rest;  // zeroed bytes, other bytes
};
Share share_of(const emu_gemm_desc_t& d, int p, bool one) {
  Share s;
  s.L = tri_layout(d.m, d.n, d.k, p, one ? 1 : 0);
  const size_t m = static_cast<size_t>(d.m), n = static_cast<size_t>(d.n);
  s.zero = al256(8 * m) + al256(8 * n) + al256(4 * p * m) + al256(4 * p * n);
  const size_t vec = 2 * static_cast<size_t>(tri_num_planes(p)) * static_cast<size_t>(s.L.kpad);
  s.rest = al256(4 * m) + al256(4 * n) + al256(vec * m) + al256(vec * n) + al256(s.L.Cs_bytes);
  return s;
}

// A batch's workspace beyond this keeps the mma.sync kernels (a fifth of it).
constexpr size_t kGroupTriBytes = size_t{32} << 30;

bool batch_one(int count, const emu_gemm_desc_t* d, int p) {
  int64_t tiles = 0;
  for (int i = 0; i < count; ++i) tiles += ((d[i].m + kBM - 1) / kBM) * ((d[i].n + kBN - 1) / kBN);
  return tiles * plan_of(p, false).nunits < 4 * kSms;
}

}  // namespace

// Batches of many small products of short K: each of their tiles is an item
// with its own chain of table loads, TMA and drain whatever it holds, and
// their int32 planes cost more than their products.  INT8 mma.sync against
// bf16 planes, us, `count` products of n x n x K:
//   p = 8, 3000: n = 32, K = 32 533 / 844, 64 603 / 862, 256 1309 / 1560; n = 64,
//     K = 32 880 / 1389, 64 1094 / 1422, 256 2625 / 2490; n = 128, K = 32 2287 /
//     3015, 64 3003 / 3090; 512: n = 256, K = 32 1345 / 1506, 64 1807 / 1518
//   p = 8, n = 16, K = 32, 512 106 / 113, 3000 504 / 684
//   p = 6, 3000: n = 32, K = 64 508 / 640, 256 1060 / 1075; n = 128, K = 32 1838 /
//     2294, 64 2284 / 2330; 512: n = 16, K = 64 101 / 86; 64: n = 64, K = 32 47 / 43
//   p = 4, 3000: n = 64, K = 32 657 / 719, 64 744 / 737; n = 16, K = 32 397 / 335
// K is the mean over the outputs; the fill is the mean outputs per 128 x 256
// tile; the lines in items per SM are where the fixed cost of a launch ends.
static bool group_tri_pays(int count, const emu_gemm_desc_t* d, int p) {
  double outs = 0.0, ks = 0.0;
  int64_t tiles = 0;
  for (int i = 0; i < count; ++i) {
    const double o = static_cast<double>(d[i].m) * static_cast<double>(d[i].n);
    outs += o;
    ks += o * static_cast<double>((d[i].k + 31) / 32 * 32);
    tiles += ((d[i].m + kBM - 1) / kBM) * ((d[i].n + kBN - 1) / kBN);
  }
  if (tiles == 0 || outs == 0.0) return true;
  const double k = ks / outs, fill = outs / static_cast<double>(tiles);
  const int64_t items = tiles * plan_of(p, false).nunits;
  if (k > 64.0) return true;
  if (fill < 500.0) return items < (p < 7 ? 200 : 100) * kSms;
  return p < 5 || items < 30 * kSms || k * fill > 1048576.0;
}

bool group_tri_takes(int count, const emu_gemm_desc_t* d, int p) {
  size_t bytes = 0;
  if (!group_tri_pays(count, d, p)) return false;
  const bool one = batch_one(count, d, p);
  for (int i = 0; i < count; ++i) {
    if (!tri_can(d[i].m, d[i].n, d[i].k, p)) return false;
    const Share s = share_of(d[i], p, one);
    bytes += s.zero + s.rest;
    if (s.L.nkc > 255 || bytes > kGroupTriBytes) return false;
  }
  return true;
}

void group_tri_free(GroupTri* g) {
  if (!g) return;
  if (g->dev) cudaFree(g->dev);
  delete g;
}

emu_status_t group_tri_build(emu_handle_s* h, int count, const emu_gemm_desc_t* d, int p, GroupTri* g) {
  g->p = p;
  g->count = count;
  g->num_sms = h->num_sms;
  g->one = batch_one(count, d, p);
  const TriPlan& tp = plan_of(p, g->one);
  std::vector<Share> sh(count);
  std::vector<int> st(3 * (count + 1), 0);
  int *sA = st.data(), *sB = sA + count + 1, *sC = sB + count + 1;
  size_t zero = 0, rest = 0;
  // items of one product and one unit length, longest first
  struct Run {
    int64_t cost;
    int prob, unit;
  };
  std::vector<Run> runs;
  for (int i = 0; i < count; ++i) {
    sh[i] = share_of(d[i], p, g->one);
    zero += sh[i].zero;
    rest += sh[i].rest;
    const TriLayout& L = sh[i].L;
    const int64_t nrun = ((L.kpad + 127) / 128 + kSplitRun - 1) / kSplitRun;
    sA[i + 1] = sA[i] + static_cast<int>((d[i].m + 7) / 8 * nrun);
    sB[i + 1] = sB[i] + static_cast<int>((d[i].n + 31) / 32 * nrun);
    sC[i + 1] = sC[i] + static_cast<int>(L.tiles_m * L.tiles_n * patch_rows(d[i].m) * patch_cols(d[i].n));
    for (int u = 0; u < tp.nunits; ++u) {
      const int64_t cols = std::min<int64_t>((d[i].n + 31) / 32 * 32, kBN);
      runs.push_back({tp.unit[u].count * L.kcs * (kBM + cols), i, u});
      g->nitems += L.nkc * L.tiles_m * L.tiles_n;
    }
  }
  std::stable_sort(runs.begin(), runs.end(), [](const Run& a, const Run& b) { return a.cost > b.cost; });
  std::vector<int4> items;
  items.reserve(static_cast<size_t>(g->nitems));
  for (const Run& r : runs) {
    const TriLayout& L = sh[r.prob].L;
    for (int kc = 0; kc < L.nkc; ++kc)
      for (int tn = 0; tn < L.tiles_n; ++tn)
        for (int tm = 0; tm < L.tiles_m; ++tm) items.push_back(make_int4(r.prob, r.unit | kc << 8, tm, tn));
  }
  g->split_blocks = sA[count] + sB[count];
  g->comb_blocks = sC[count];
  size_t off = 0;
  const size_t o_probs = off; off += al256(sizeof(GTriProb) * count);
  const size_t o_maps = off; off += al256(sizeof(CUtensorMap) * 2 * count);
  const size_t o_items = off; off += al256(sizeof(int4) * items.size());
  const size_t o_st = off; off += al256(sizeof(int) * st.size());
  const size_t o_zero = off; off += zero;
  const size_t o_rest = off; off += rest;
  if (cudaMalloc(&g->dev, off) != cudaSuccess) {
    g->dev = nullptr;
    cudaGetLastError();
    return EMU_ERR_ALLOC;
  }
  uint8_t* const base = static_cast<uint8_t*>(g->dev);
  g->d_probs = reinterpret_cast<GTriProb*>(base + o_probs);
  g->d_maps = reinterpret_cast<CUtensorMap*>(base + o_maps);
  g->d_items = reinterpret_cast<int4*>(base + o_items);
  g->d_startA = reinterpret_cast<int*>(base + o_st);
  g->d_startB = g->d_startA + count + 1;
  g->d_startC = g->d_startB + count + 1;
  g->zero = base + o_zero;
  g->zero_bytes = zero;
  uint8_t *pz = base + o_zero, *pr = base + o_rest;
  auto take = [](uint8_t*& at, size_t bytes) {
    uint8_t* const p0 = at;
    at += al256(bytes);
    return p0;
  };
  std::vector<GTriProb> probs(count);
  std::vector<CUtensorMap> maps(2 * count);
  const int np = tri_num_planes(p);
  for (int i = 0; i < count; ++i) {
    const TriLayout& L = sh[i].L;
    GTriProb& q = probs[i];
    const size_t m = static_cast<size_t>(d[i].m), n = static_cast<size_t>(d[i].n);
    const size_t vec = 2 * static_cast<size_t>(np) * static_cast<size_t>(L.kpad);
    q.A = d[i].A;
    q.B = d[i].B;
    q.C = d[i].C;
    q.lda = d[i].lda;
    q.ldb = d[i].ldb;
    q.ldc = d[i].ldc;
    q.kpad = L.kpad;
    q.alpha = d[i].alpha;
    q.beta = d[i].beta;
    q.maxA = reinterpret_cast<unsigned long long*>(take(pz, 8 * m));
    q.maxB = reinterpret_cast<unsigned long long*>(take(pz, 8 * n));
    q.sumA = reinterpret_cast<int32_t*>(take(pz, 4 * p * m));
    q.sumB = reinterpret_cast<int32_t*>(take(pz, 4 * p * n));
    q.EA = reinterpret_cast<int32_t*>(take(pr, 4 * m));
    q.FB = reinterpret_cast<int32_t*>(take(pr, 4 * n));
    q.planesA = reinterpret_cast<uint16_t*>(take(pr, vec * m));
    q.planesB = reinterpret_cast<uint16_t*>(take(pr, vec * n));
    q.Cs = reinterpret_cast<int32_t*>(take(pr, L.Cs_bytes));
    tri_const(p, d[i].k, &q.const_lo, &q.const_hi);
    q.M = static_cast<int>(m);
    q.N = static_cast<int>(n);
    q.K = static_cast<int>(d[i].k);
    q.nst = static_cast<int>(L.kpad / 64);
    q.kcs = static_cast<int>(L.kcs);
    q.nkc = static_cast<int>(L.nkc);
    q.tiles_m = static_cast<int>(L.tiles_m);
    q.tiles_n = static_cast<int>(L.tiles_n);
    // boxes no higher than the product (rows in steps of the 8-row swizzle atoms)
    const uint32_t ra = static_cast<uint32_t>(std::min<size_t>((m + 7) / 8 * 8, kBM));
    const uint32_t rb = static_cast<uint32_t>(std::min<size_t>((n + 31) / 32 * 32, kBN));
    q.box_bytes = static_cast<int>((ra + rb) * 128);
    if (!make_tmap_i8(&maps[2 * i], q.planesA, 2 * static_cast<uint64_t>(L.kpad), m * np, ra, 128) ||
        !make_tmap_i8(&maps[2 * i + 1], q.planesB, 2 * static_cast<uint64_t>(L.kpad), n * np, rb, 128))
      return EMU_ERR_CUDA;
    g->maxA.push_back(q.maxA);
    g->maxB.push_back(q.maxB);
  }
  const bool ok =
      cudaMemcpy(g->d_probs, probs.data(), sizeof(GTriProb) * count, cudaMemcpyHostToDevice) == cudaSuccess &&
      cudaMemcpy(g->d_maps, maps.data(), sizeof(CUtensorMap) * 2 * count, cudaMemcpyHostToDevice) == cudaSuccess &&
      cudaMemcpy(g->d_items, items.data(), sizeof(int4) * items.size(), cudaMemcpyHostToDevice) == cudaSuccess &&
      cudaMemcpy(g->d_startA, st.data(), sizeof(int) * st.size(), cudaMemcpyHostToDevice) == cudaSuccess;
  return ok ? EMU_OK : EMU_ERR_CUDA;
}

cudaError_t group_tri_prepare() {
  return cudaFuncSetAttribute(gemm_I_grouped_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              bf16g::Cfg<false>::kSmem);
}

template <int P>
static cudaError_t launch_p(const GroupTri& g, int* status, cudaStream_t st) {
  grouped_split_tri_kernel<P><<<g.split_blocks, 256, 0, st>>>(g.d_probs, g.count, g.d_startA, g.d_startB);
  KParamsGTri kp;
  kp.tp = plan_of(P, g.one);
  kp.probs = g.d_probs;
  kp.maps = g.d_maps;
  kp.items = g.d_items;
  kp.nitems = static_cast<int>(g.nitems);
  kp.status = status;
  const int grid = static_cast<int>(std::min<int64_t>(g.nitems, g.num_sms));
  gemm_I_grouped_tc_kernel<<<grid, bf16g::kThreads, bf16g::Cfg<false>::kSmem, st>>>(kp);
  if (g.one)
    grouped_combine_kernel<P, true><<<g.comb_blocks, 256, 0, st>>>(g.d_probs, g.count, g.d_startC);
  else
    grouped_combine_kernel<P, false><<<g.comb_blocks, 256, 0, st>>>(g.d_probs, g.count, g.d_startC);
  return cudaGetLastError();
}

cudaError_t group_tri_launch(const GroupTri& g, int* status, cudaStream_t st) {
  switch (g.p) {
#define EMU_CASE(PP) \
  case PP:           \
    return launch_p<PP>(g, status, st);
    EMU_CASE(1) EMU_CASE(2) EMU_CASE(3) EMU_CASE(4) EMU_CASE(5) EMU_CASE(6) EMU_CASE(7) EMU_CASE(8)
#undef EMU_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace emu
