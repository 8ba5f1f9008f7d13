// select.cu -- learned slice-count selector for Scheme I (auto precision).
//
// The paper picks p by hand and notes that it lacks an automatic precision
// choice (Sec. VII).  This file adds one: per-product features (exponent
// deficit histograms of sampled rows of A and columns of B, log2 k and the
// requested tolerance), a 66-64-64-8 MLP with hand-written FP32 forward,
// backward and Adam kernels, a double-double probe of sampled output entries
// that judges a prediction, and emu_dgemm_auto, which escalates p when the
// probe finds the tolerance missed.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include <cooperative_groups.h>

#include "emu_handle.h"
#include "emu_internal.h"

namespace cg = cooperative_groups;

namespace emu {

namespace {

constexpr int kIn = EMU_SEL_IN, kHid = EMU_SEL_HID, kOut = EMU_SEL_OUT;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kHid * kIn, kOffW2 = kOffB1 + kHid, kOffB2 = kOffW2 + kHid * kHid,
              kOffW3 = kOffB2 + kHid, kOffB3 = kOffW3 + kOut * kHid, kNParam = kOffB3 + kOut;
static_assert(kNParam == EMU_SEL_NPARAM, "parameter count");

struct SelState {
  float* params = nullptr;  // device, loaded weights (Scheme I: classes p = 3..10)
  bool loaded = false;
  float* params_II = nullptr;  // Scheme II, norm scaling: classes N = 6, 8, .., 20
  bool loaded_II = false;
  // auto-precision buffers, grown on demand (layout: auto_impl): device
  // memory, and pinned host memory that the kernels write their few results
  // into
  uint8_t* dev = nullptr;
  size_t dev_bytes = 0;
  uint8_t* host = nullptr;
  size_t host_bytes = 0;
  // side stream for the probe's reference sums (they depend on A and B only,
  // so they run beside the product)
  cudaStream_t side = nullptr;
  cudaEvent_t ev_decide = nullptr, ev_fork = nullptr, ev_probe = nullptr;
};
SelState* sel_of(emu_handle_s* h) {
  if (!h->selector) h->selector = new SelState();
  return static_cast<SelState*>(h->selector);
}

// ---------------------------------------------------------------- features
// Exponent of |x| from its bits: frexp exponent (E with |x| in [2^(E-1), 2^E)).
__device__ __forceinline__ int exp_bits(uint64_t ab) { return frexp_exp_bits(ab); }

// One block per sampled vector: 32-bin histogram of the exponent deficit
// d = E_vec - e(x) in bins of 3 exponents (bin = min(d / 3, 31); x == 0 ->
// bin 31), added to hist (uint32[32]).  E_vec, the exponent of the vector's
// largest magnitude, is found by the block first (the vector is then read
// a second time, from L2), so that no pass over the whole of A and B is
// needed for 64 sampled vectors.
// One launch serves both operands: blocks [0, nblk_a) sample A (histogram
// hist[0..31]), the rest sample B (hist[32..63]).
struct FeatOperand {
  const double* X;
  int64_t ld;
  bool kcontig;
  int64_t rows, stride;
};
// The block that finishes last turns the histograms into the features and,
// with a network loaded (prm), its class probabilities: one launch decides.
// It is latency bound (a few microseconds of dependent loads), so there is no
// second and third kernel, and the results go straight to `out` (feat[128 |
// prob], pinned host memory in the auto entry points, beside the device copy
// `feat`), which spares the copy back.  The histograms and the counter are
// zero before and after the launch.
struct FeatDecide {
  unsigned int* done;  // blocks-finished counter
  float log2k_16, ltol_16;
  const float* prm;  // null: features only
  float* feat;       // device, 66 floats
  float* out;        // null: no second copy; else features at 0, probabilities at 128
  uint4* zero;  // nzero 16-byte words to zero
  int64_t nzero;
};
__device__ void feat_decide(const FeatDecide& d, unsigned int* hist);
__global__ void __launch_bounds__(256) feat_hist_kernel(FeatOperand oa, FeatOperand ob, int nblk_a, int64_t k,
                                                        unsigned int* __restrict__ hist_all, FeatDecide dec) {
  __shared__ unsigned int sh[32];
  __shared__ unsigned long long wmax[8];
  if (threadIdx.x < 32) sh[threadIdx.x] = 0;
  // (what the scan and the split after it add to, zeroed on the way)
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; i < dec.nzero; i += 256 * gridDim.x)
    dec.zero[i] = make_uint4(0, 0, 0, 0);
  const bool is_a = static_cast<int>(blockIdx.x) < nblk_a;
  const FeatOperand& op = is_a ? oa : ob;
  unsigned int* __restrict__ hist = hist_all + (is_a ? 0 : 32);
  const int64_t r = static_cast<int64_t>(is_a ? blockIdx.x : blockIdx.x - nblk_a) * op.stride;
  const bool live = r < op.rows;
  const double* const p = op.kcontig ? op.X + r * op.ld : op.X + r;
  const int64_t sp = op.kcontig ? 1 : op.ld;
  auto absbits = [&](int64_t h) { return dbits(__ldg(p + h * sp)) & 0x7FFFFFFFFFFFFFFFull; };
  // the first kFeatReg x 256 elements of the vector stay in registers between
  // the two passes, the rest is read twice
  constexpr int kFeatReg = 12;
  unsigned long long v[kFeatReg];
  unsigned long long mx = 0;  // largest |x| bit pattern (NaN > inf > finite)
#pragma unroll
  for (int q = 0; q < kFeatReg; ++q) {
    const int64_t h = threadIdx.x + 256 * q;
    v[q] = live && h < k ? absbits(h) : 0;
  }
#pragma unroll
  for (int q = 0; q < kFeatReg; ++q) mx = v[q] > mx ? v[q] : mx;
  if (live)
    for (int64_t h = threadIdx.x + 256 * kFeatReg; h < k; h += 256) {
      const unsigned long long ab = absbits(h);
      mx = ab > mx ? ab : mx;
    }
  for (int o = 16; o; o >>= 1) {
    const unsigned long long other = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = other > mx ? other : mx;
  }
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (live) {
    uint64_t mb = wmax[0];
#pragma unroll
    for (int q = 1; q < 8; ++q) mb = wmax[q] > mb ? wmax[q] : mb;
    const int E = mb >= 0x7FF0000000000000ull ? 0 : exp_bits(mb);
    // most elements of a vector share a few bins: one add per warp and bin
    auto count = [&](uint64_t ab) {
      int bin = 31;
      if (ab != 0 && ab < 0x7FF0000000000000ull) {
        const int d = E - exp_bits(ab);
        bin = d < 0 ? 0 : (d / 3 > 31 ? 31 : d / 3);
      }
      const unsigned same = __match_any_sync(__activemask(), bin);
      if ((threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&sh[bin], static_cast<unsigned>(__popc(same)));
    };
#pragma unroll
    for (int q = 0; q < kFeatReg; ++q)
      if (threadIdx.x + 256 * q < k) count(v[q]);
    for (int64_t h = threadIdx.x + 256 * kFeatReg; h < k; h += 256) count(absbits(h));
  }
  __syncthreads();
  if (threadIdx.x < 32 && sh[threadIdx.x]) atomicAdd(&hist[threadIdx.x], sh[threadIdx.x]);
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(dec.done, 1u) + 1 == gridDim.x;
  __syncthreads();
  if (!last) return;
  __threadfence();
  feat_decide(dec, hist_all);
}

// The last block (256 threads) of feat_hist_kernel.
__device__ void feat_decide(const FeatDecide& d, unsigned int* hist) {
  __shared__ unsigned int hs[64];
  __shared__ float x[kIn + 2], h1[kHid], h2[kHid], z[kOut], tot[2];
  const int t = threadIdx.x;
  // each neuron's weights to its thread's registers, all loads in flight
  // together (66 and 64 of them one after another were most of the time)
  float2 w1[kIn / 2];
  float4 w2[kHid / 4], w3[kHid / 4];
  float b1 = 0.f, b2 = 0.f, b3 = 0.f;
  static_assert(kIn % 2 == 0 && kHid % 4 == 0 && kOffW2 % 4 == 0 && kOffW3 % 4 == 0, "vector loads of the weights");
  if (d.prm && t < kHid) {
    const float* r1 = d.prm + kOffW1 + t * kIn;
    const float* r2 = d.prm + kOffW2 + t * kHid;
    const float* r3 = d.prm + kOffW3 + (t < kOut ? t : 0) * kHid;
#pragma unroll
    for (int i = 0; i < kIn / 2; ++i) w1[i] = __ldg(reinterpret_cast<const float2*>(r1) + i);
#pragma unroll
    for (int i = 0; i < kHid / 4; ++i) w2[i] = __ldg(reinterpret_cast<const float4*>(r2) + i);
#pragma unroll
    for (int i = 0; i < kHid / 4; ++i) w3[i] = __ldg(reinterpret_cast<const float4*>(r3) + i);
    b1 = __ldg(d.prm + kOffB1 + t);
    b2 = __ldg(d.prm + kOffB2 + t);
    b3 = __ldg(d.prm + kOffB3 + (t < kOut ? t : 0));
  }
  if (t < 64) {
    hs[t] = __ldcg(hist + t);
    hist[t] = 0;
  }
  if (t == 64) *d.done = 0;
  __syncthreads();
  if (t < 2) {
    unsigned int s = 0;
    for (int i = 0; i < 32; ++i) s += hs[t * 32 + i];
    tot[t] = s ? static_cast<float>(s) : 1.0f;
  }
  __syncthreads();
  if (t < kIn) {
    const float f = t < 64 ? static_cast<float>(hs[t]) / tot[t / 32] : t == 64 ? d.log2k_16 : d.ltol_16;
    x[t] = f;
    d.feat[t] = f;
    if (d.out) d.out[t] = f;
  }
  if (!d.prm) return;
  __syncthreads();
  // the arithmetic of mlp_forward_kernel, in its order
  auto dot4 = [](const float4* w, const float* v, float s) {
#pragma unroll
    for (int i = 0; i < kHid / 4; ++i) {
      s = fmaf(w[i].x, v[4 * i], s);
      s = fmaf(w[i].y, v[4 * i + 1], s);
      s = fmaf(w[i].z, v[4 * i + 2], s);
      s = fmaf(w[i].w, v[4 * i + 3], s);
    }
    return s;
  };
  if (t < kHid) {
    float s = b1;
#pragma unroll
    for (int i = 0; i < kIn / 2; ++i) {
      s = fmaf(w1[i].x, x[2 * i], s);
      s = fmaf(w1[i].y, x[2 * i + 1], s);
    }
    h1[t] = s > 0.f ? s : 0.f;
  }
  __syncthreads();
  if (t < kHid) {
    const float s = dot4(w2, h1, b2);
    h2[t] = s > 0.f ? s : 0.f;
  }
  __syncthreads();
  if (t < kOut) z[t] = dot4(w3, h2, b3);
  __syncthreads();
  if (t < kOut) {
    float mx = z[0];
    for (int o = 1; o < kOut; ++o) mx = fmaxf(mx, z[o]);
    float den = 0.f;
    for (int o = 0; o < kOut; ++o) den += expf(z[o] - mx);
    d.out[128 + t] = expf(z[t] - mx) / den;
  }
}

// ---------------------------------------------------------------- MLP
// One block of 64 threads per sample.  act (optional): [h1 | h2] per sample.
__global__ void mlp_forward_kernel(const float* __restrict__ prm, const float* __restrict__ X, int64_t batch,
                                   float* __restrict__ P, float* __restrict__ act) {
  __shared__ float x[kIn], h1[kHid], h2[kHid], z[kOut];
  const int64_t b = blockIdx.x;
  const int j = threadIdx.x;
  if (b >= batch) return;
  for (int i = j; i < kIn; i += blockDim.x) x[i] = X[b * kIn + i];
  __syncthreads();
  float s = prm[kOffB1 + j];
  for (int i = 0; i < kIn; ++i) s = fmaf(prm[kOffW1 + j * kIn + i], x[i], s);
  h1[j] = s > 0.f ? s : 0.f;
  __syncthreads();
  s = prm[kOffB2 + j];
  for (int i = 0; i < kHid; ++i) s = fmaf(prm[kOffW2 + j * kHid + i], h1[i], s);
  h2[j] = s > 0.f ? s : 0.f;
  __syncthreads();
  if (j < kOut) {
    float t = prm[kOffB3 + j];
    for (int i = 0; i < kHid; ++i) t = fmaf(prm[kOffW3 + j * kHid + i], h2[i], t);
    z[j] = t;
  }
  __syncthreads();
  if (j < kOut) {
    float mx = z[0];
    for (int o = 1; o < kOut; ++o) mx = fmaxf(mx, z[o]);
    float den = 0.f;
    for (int o = 0; o < kOut; ++o) den += expf(z[o] - mx);
    P[b * kOut + j] = expf(z[j] - mx) / den;
  }
  if (act) {
    act[b * 2 * kHid + j] = h1[j];
    act[b * 2 * kHid + kHid + j] = h2[j];
  }
}

// Mean cross-entropy backward.  Each block takes `per` samples, accumulates
// the parameter gradient in shared memory and adds it to grad once.
__global__ void mlp_backward_kernel(const float* __restrict__ prm, const float* __restrict__ X,
                                    const float* __restrict__ act, const float* __restrict__ P,
                                    const int32_t* __restrict__ y, int64_t batch, int per, float* __restrict__ grad,
                                    float* __restrict__ loss) {
  extern __shared__ float g[];  // kNParam floats
  __shared__ float dz[kOut], dh2[kHid], dh1[kHid];
  const int j = threadIdx.x;  // 64 threads
  for (int i = j; i < kNParam; i += blockDim.x) g[i] = 0.f;
  __syncthreads();
  const float inv = 1.0f / static_cast<float>(batch);
  float lsum = 0.f;
  for (int q = 0; q < per; ++q) {
    int64_t b = static_cast<int64_t>(blockIdx.x) * per + q;
    if (b >= batch) break;
    const float* x = X + b * kIn;
    const float* h1 = act + b * 2 * kHid;
    const float* h2 = h1 + kHid;
    const int lab = y[b];
    if (j < kOut) dz[j] = (P[b * kOut + j] - (j == lab ? 1.f : 0.f)) * inv;
    if (j == 0) lsum += -logf(fmaxf(P[b * kOut + lab], 1e-30f));
    __syncthreads();
    // layer 3
    for (int o = 0; o < kOut; ++o) g[kOffW3 + o * kHid + j] += dz[o] * h2[j];
    if (j < kOut) g[kOffB3 + j] += dz[j];
    float s = 0.f;
    for (int o = 0; o < kOut; ++o) s = fmaf(prm[kOffW3 + o * kHid + j], dz[o], s);
    dh2[j] = h2[j] > 0.f ? s : 0.f;
    __syncthreads();
    // layer 2 (thread j owns row j of W2)
    for (int i = 0; i < kHid; ++i) g[kOffW2 + j * kHid + i] += dh2[j] * h1[i];
    g[kOffB2 + j] += dh2[j];
    s = 0.f;
    for (int o = 0; o < kHid; ++o) s = fmaf(prm[kOffW2 + o * kHid + j], dh2[o], s);
    dh1[j] = h1[j] > 0.f ? s : 0.f;
    __syncthreads();
    // layer 1 (thread j owns row j of W1)
    for (int i = 0; i < kIn; ++i) g[kOffW1 + j * kIn + i] += dh1[j] * x[i];
    g[kOffB1 + j] += dh1[j];
    __syncthreads();
  }
  for (int i = j; i < kNParam; i += blockDim.x)
    if (g[i] != 0.f) atomicAdd(&grad[i], g[i]);
  if (j == 0 && lsum != 0.f) atomicAdd(loss, lsum * inv);
}

__global__ void adam_kernel(float* __restrict__ prm, const float* __restrict__ grad, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float gi = grad[i];
  float mi = b1 * m[i] + (1.f - b1) * gi;
  float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  prm[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ---------------------------------------------------------------- probe
struct DD {
  double hi, lo;
};
__device__ __forceinline__ DD dd_add(DD a, DD b) {
  double s = __dadd_rn(a.hi, b.hi);
  double z = __dsub_rn(s, a.hi);
  double e = __dadd_rn(__dsub_rn(a.hi, __dsub_rn(s, z)), __dsub_rn(b.hi, z));
  e = __dadd_rn(e, __dadd_rn(a.lo, b.lo));
  double t = __dadd_rn(s, e);
  return {t, __dsub_rn(e, __dsub_rn(t, s))};
}

// Per sampled entry (i, j) a cluster of eight one-warp blocks: compensated
// dot product (TwoProduct by fma, TwoSum accumulation) per thread over a
// strided share of K (256 threads per entry), threads combined by
// double-double adds (warp shuffles, then the warps' partial results through
// the first block's shared memory).  FP64 issue bounds it (two results per
// clock and SM), and it runs beside the product whose persistent GEMM wants
// every SM: eight warps of one block on each of 64 SMs held those SMs back,
// 64 x 8 single warps spread over the whole GPU do not.
constexpr int kProbeWarps = 8, kProbeThreads = 32 * kProbeWarps;
__global__ void __cluster_dims__(kProbeWarps, 1, 1) __launch_bounds__(32)
    probe_dd_kernel(const double* __restrict__ A, int64_t lda, bool a_kcontig, const double* __restrict__ B,
                    int64_t ldb, bool b_kcontig, int64_t k, int count, const int32_t* __restrict__ idx,
                    double* __restrict__ ref, double* __restrict__ absab) {
  __shared__ double sh[3][kProbeWarps];
  cg::cluster_group cl = cg::this_cluster();
  const int w = blockIdx.x / kProbeWarps, lane = threadIdx.x, wp = blockIdx.x % kProbeWarps;
  const int64_t i = idx[2 * w], j = idx[2 * w + 1];
  const double* const pa = a_kcontig ? A + i * lda : A + i;
  const double* const pb = b_kcontig ? B + j * ldb : B + j;
  const int64_t sa = a_kcontig ? 1 : lda, sb = b_kcontig ? 1 : ldb;
  DD acc{0.0, 0.0};
  double ab = 0.0;
#pragma unroll 4
  for (int64_t h = wp * 32 + lane; h < k; h += kProbeThreads) {
    const double a = __ldg(pa + h * sa);
    const double b = __ldg(pb + h * sb);
    const double p = __dmul_rn(a, b);
    const double e = __fma_rn(a, b, -p);
    acc = dd_add(acc, DD{p, e});
    ab = __fma_rn(fabs(a), fabs(b), ab);
  }
  for (int o = 16; o; o >>= 1) {
    DD other{__shfl_xor_sync(0xffffffffu, acc.hi, o), __shfl_xor_sync(0xffffffffu, acc.lo, o)};
    acc = dd_add(acc, other);
    ab = __dadd_rn(ab, __shfl_xor_sync(0xffffffffu, ab, o));
  }
  cl.sync();  // the first block runs: its shared memory may be written
  if (lane == 0) {
    double* dst = cl.map_shared_rank(&sh[0][0], 0);
    dst[wp] = acc.hi;
    dst[kProbeWarps + wp] = acc.lo;
    dst[2 * kProbeWarps + wp] = ab;
  }
  cl.sync();
  if (wp == 0 && lane == 0) {
    DD t{sh[0][0], sh[1][0]};
    double tab = sh[2][0];
    for (int q = 1; q < kProbeWarps; ++q) {
      t = dd_add(t, DD{sh[0][q], sh[1][q]});
      tab = __dadd_rn(tab, sh[2][q]);
    }
    ref[2 * w] = t.hi;
    ref[2 * w + 1] = t.lo;
    absab[w] = tab;
  }
}

// Probe entries: a deterministic spread over C (caller's coordinates), the
// xorshift sequence from the shape.
__global__ void probe_idx_kernel(uint64_t x, int64_t m, int64_t n, int count, int32_t* __restrict__ idx) {
  for (int q = 0; q < 2 * count; ++q) {
    x ^= x << 13;
    x ^= x >> 7;
    x ^= x << 17;
    idx[q] = static_cast<int32_t>(x % static_cast<uint64_t>(q & 1 ? n : m));
  }
}

// The probed entries of C with their reference sums, to pinned host memory:
// out = [ref (hi, lo) | sum |a||b| | C entry], `count` of each.  idx holds
// the caller's (i, j); colmajor: C's rows are the caller's columns.
__global__ void __launch_bounds__(256) judge_kernel(const double* __restrict__ C, int64_t ldc, bool colmajor,
                                                    int count, const int32_t* __restrict__ idx,
                                                    const double* __restrict__ ref, const double* __restrict__ ab,
                                                    double* __restrict__ out) {
  for (int w = threadIdx.x; w < count; w += 256) {
    const int64_t i = idx[2 * w], j = idx[2 * w + 1];
    out[2 * w] = ref[2 * w];
    out[2 * w + 1] = ref[2 * w + 1];
    out[2 * static_cast<int64_t>(count) + w] = ab[w];
    out[3 * static_cast<int64_t>(count) + w] = C[colmajor ? j * ldc + i : i * ldc + j];
  }
}

}  // namespace

void selector_release(emu_handle_s* h) {
  auto* s = static_cast<SelState*>(h->selector);
  if (!s) return;
  if (s->params) cudaFree(s->params);
  if (s->params_II) cudaFree(s->params_II);
  if (s->dev) cudaFree(s->dev);
  if (s->host) cudaFreeHost(s->host);
  if (s->side) cudaStreamDestroy(s->side);
  if (s->ev_fork) cudaEventDestroy(s->ev_fork);
  if (s->ev_decide) cudaEventDestroy(s->ev_decide);
  if (s->ev_probe) cudaEventDestroy(s->ev_probe);
  delete s;
  h->selector = nullptr;
}

}  // namespace emu

using namespace emu;

namespace {

// Features of one product into feat (device float[66]); needs feat_scratch
// bytes of scratch (histograms and the blocks-finished counter; zeroed: they
// are zero already, as an earlier call leaves them).  prm: also
// the network's class probabilities; out: see FeatDecide.
emu_status_t features_impl(const View& v, int64_t k, double tol, int64_t sample, float* feat, uint8_t* scratch,
                           cudaStream_t st, bool zeroed = false, const float* prm = nullptr, float* out = nullptr, 
                           uint4* zero = nullptr, int64_t nzero = 0) {
  auto* hist = reinterpret_cast<unsigned int*>(scratch);
  if (!zeroed) cudaMemsetAsync(hist, 0, 65 * sizeof(unsigned int), st);
  int64_t sa = sample > 0 ? std::max<int64_t>(1, v.M / sample) : 1;
  int64_t sb = sample > 0 ? std::max<int64_t>(1, v.N / sample) : 1;
  int64_t na = (v.M + sa - 1) / sa, nb = (v.N + sb - 1) / sb;
  if (sample > 0) {
    na = std::min<int64_t>(na, sample);
    nb = std::min<int64_t>(nb, sample);
  }
  const FeatOperand oa{static_cast<const double*>(v.A), v.ldA, v.a_kcontig, v.M, sa};
  const FeatOperand ob{static_cast<const double*>(v.B), v.ldB, v.b_kcontig, v.N, sb};
  const FeatDecide dec{hist + 64, static_cast<float>(std::log2(static_cast<double>(k)) / 16.0),
                       static_cast<float>(-std::log10(tol) / 16.0), prm, feat, out, zero, nzero};
  feat_hist_kernel<<<static_cast<unsigned>(na + nb), 256, 0, st>>>(
      oa, ob, static_cast<int>(na), k, hist, dec);
  return cudaGetLastError() == cudaSuccess ? EMU_OK : EMU_ERR_CUDA;
}

size_t feat_scratch(const View&) { return 512; }

bool valid_layout(emu_layout_t l) { return l == EMU_ROW_MAJOR || l == EMU_COL_MAJOR; }

// Bound-based p: smallest p in [3, 10] with 2^(-8p+3) * 2^spread * k <= tol,
// spread = the upper edge of the largest exponent-deficit bin seen.
// Scheme II with norm scaling: a' = trunc(a 2^(h - e_i)) errs by less than
// 2^(e_i - h) and e_i exceeds the frexp exponent of an entry by at most the
// deficit d against the row maximum plus ceil(log2(k) / 2), so every term
// of the product errs by at most 2^(-h + d + ceil(log2(k)/2) + 3) of its
// magnitude.  Smallest N in 6, 8, .., 20 meeting tol with d = spread (20 if
// none does).  A heuristic fallback, like the Scheme I bound.
int bound_nm_from_hist(const float* f, int64_t k, double tol) {
  int spread = 0;
  for (int i = 0; i < 64; ++i)
    if (f[i] > 0.f) spread = std::max(spread, 3 * (i % 32) + 2);
  int half_lk = 0;
  while ((int64_t{1} << (2 * half_lk)) < k) ++half_lk;  // ceil(log2(k) / 2)
  for (int nm = EMU_SEL_NM0; nm <= EMU_NM_MAX; nm += 2) {
    int hA, hB;
    host_norm_halves_II(nm, &hA, &hB);
    if (std::ldexp(1.0, -hA + spread + half_lk + 3) <= tol) return nm;
  }
  return EMU_NM_MAX;
}

int bound_p_from_hist(const float* f, int64_t k, double tol) {
  int spread = 0;
  for (int i = 0; i < 64; ++i)
    if (f[i] > 0.f) spread = std::max(spread, 3 * (i % 32) + 2);
  for (int p = 3; p <= 10; ++p)
    if (std::ldexp(1.0, -8 * p + 3 + spread) * static_cast<double>(k) <= tol) return p;
  return 10;
}

// Bound-based choice (host), shared by emu_bound_p and emu_bound_nm.
emu_status_t bound_impl(emu_handle_s* h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, const double* A,
                        int64_t lda, const double* B, int64_t ldb, double tol, int* out, emu_stream_t stream,
                        bool scheme_II) {
  if (!out || !h) return EMU_ERR_INVALID_ARG;
  if ((layout != EMU_ROW_MAJOR && layout != EMU_COL_MAJOR) || m < 1 || n < 1 || k < 1 || !A || !B || !(tol > 0.0))
    return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  View v;
  normalize(layout, m, n, A, lda, B, ldb, &v);
  uint8_t* ws = nullptr;
  const size_t need = feat_scratch(v) + 512;
  emu_status_t s = handle_workspace(h, need, st, &ws);
  if (s != EMU_OK) return s;
  float* feat = reinterpret_cast<float*>(ws + feat_scratch(v));
  s = features_impl(v, k, tol, 64, feat, ws, st);
  if (s != EMU_OK) return s;
  float f[kIn];
  if (cudaMemcpyAsync(f, feat, sizeof(f), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return EMU_ERR_CUDA;
  *out = scheme_II ? bound_nm_from_hist(f, k, tol) : bound_p_from_hist(f, k, tol);
  return EMU_OK;
}

}  // namespace

extern "C" {

emu_status_t emu_sel_features(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, const double* A,
                              int64_t lda, const double* B, int64_t ldb, double tol, int64_t sample, float* feat,
                              emu_stream_t stream) {
  if (!h || !feat || !A || !B || m < 1 || n < 1 || k < 1 || !(tol > 0.0) || !valid_layout(layout))
    return EMU_ERR_INVALID_ARG;
  if (!check_lds(layout, m, n, k, lda, ldb, layout == EMU_ROW_MAJOR ? n : m)) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  View v;
  normalize(layout, m, n, A, lda, B, ldb, &v);
  uint8_t* ws = nullptr;
  emu_status_t s = handle_workspace(h, feat_scratch(v), st, &ws);
  if (s != EMU_OK) return s;
  return features_impl(v, k, tol, sample, feat, ws, st);
}

emu_status_t emu_sel_forward(emu_handle_t h, int64_t batch, const float* prm, const float* X, float* P, float* act,
                             emu_stream_t stream) {
  if (!h || !prm || !X || !P || batch < 0) return EMU_ERR_INVALID_ARG;
  if (batch == 0) return EMU_OK;
  if (batch > INT32_MAX) return EMU_ERR_UNSUPPORTED;
  cudaSetDevice(h->device);
  mlp_forward_kernel<<<static_cast<unsigned>(batch), kHid, 0, static_cast<cudaStream_t>(stream)>>>(prm, X, batch, P,
                                                                                                    act);
  return cudaGetLastError() == cudaSuccess ? EMU_OK : EMU_ERR_CUDA;
}

emu_status_t emu_sel_backward(emu_handle_t h, int64_t batch, const float* prm, const float* X, const float* act,
                              const float* P, const int32_t* y, float* grad, float* loss, emu_stream_t stream) {
  if (!h || !prm || !X || !act || !P || !y || !grad || !loss || batch < 1) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int per = 32;
  const int smem = kNParam * static_cast<int>(sizeof(float));
  if (cudaFuncSetAttribute(mlp_backward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
    return EMU_ERR_CUDA;
  cudaMemsetAsync(grad, 0, sizeof(float) * kNParam, st);
  cudaMemsetAsync(loss, 0, sizeof(float), st);
  unsigned blocks = static_cast<unsigned>((batch + per - 1) / per);
  mlp_backward_kernel<<<blocks, kHid, smem, st>>>(prm, X, act, P, y, batch, per, grad, loss);
  return cudaGetLastError() == cudaSuccess ? EMU_OK : EMU_ERR_CUDA;
}

emu_status_t emu_sel_adam(emu_handle_t h, float* prm, const float* grad, float* m, float* v, int step, float lr,
                          float b1, float b2, float eps, emu_stream_t stream) {
  if (!h || !prm || !grad || !m || !v || step < 1) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  float c1 = 1.f - std::pow(b1, static_cast<float>(step)), c2 = 1.f - std::pow(b2, static_cast<float>(step));
  adam_kernel<<<(kNParam + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(prm, grad, m, v, kNParam, lr, b1,
                                                                                      b2, eps, c1, c2);
  return cudaGetLastError() == cudaSuccess ? EMU_OK : EMU_ERR_CUDA;
}

emu_status_t emu_sel_load(emu_handle_t h, const float* params) {
  if (!h || !params) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  SelState* s = sel_of(h);
  if (!s->params && cudaMalloc(&s->params, sizeof(float) * kNParam) != cudaSuccess) return EMU_ERR_ALLOC;
  if (cudaMemcpy(s->params, params, sizeof(float) * kNParam, cudaMemcpyHostToDevice) != cudaSuccess)
    return EMU_ERR_CUDA;
  s->loaded = true;
  return EMU_OK;
}

emu_status_t emu_sel_load_II(emu_handle_t h, const float* params) {
  if (!h || !params) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  SelState* s = sel_of(h);
  if (!s->params_II && cudaMalloc(&s->params_II, sizeof(float) * kNParam) != cudaSuccess) return EMU_ERR_ALLOC;
  if (cudaMemcpy(s->params_II, params, sizeof(float) * kNParam, cudaMemcpyHostToDevice) != cudaSuccess)
    return EMU_ERR_CUDA;
  s->loaded_II = true;
  return EMU_OK;
}

emu_status_t emu_probe_dd(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, const double* A,
                          int64_t lda, const double* B, int64_t ldb, int count, const int32_t* idx, double* ref,
                          double* absab, emu_stream_t stream) {
  if (!h || !A || !B || !idx || !ref || !absab || count < 0 || m < 1 || n < 1 || k < 1 || !valid_layout(layout))
    return EMU_ERR_INVALID_ARG;
  if (!check_lds(layout, m, n, k, lda, ldb, layout == EMU_ROW_MAJOR ? n : m)) return EMU_ERR_INVALID_ARG;
  if (count == 0) return EMU_OK;
  cudaSetDevice(h->device);
  // entries are given in the caller's (i, j) of C; the kernel reads A rows
  // and B columns directly in the caller's layout
  bool a_k = layout == EMU_ROW_MAJOR, b_k = layout != EMU_ROW_MAJOR;
  probe_dd_kernel<<<count * kProbeWarps, 32, 0, static_cast<cudaStream_t>(stream)>>>(A, lda, a_k, B, ldb, b_k, k,
                                                                                 count, idx, ref, absab);
  return cudaGetLastError() == cudaSuccess ? EMU_OK : EMU_ERR_CUDA;
}

emu_status_t emu_bound_p(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, const double* A,
                         int64_t lda, const double* B, int64_t ldb, double tol, int* p_out, emu_stream_t stream) {
  return bound_impl(h, layout, m, n, k, A, lda, B, ldb, tol, p_out, stream, false);
}

emu_status_t emu_bound_nm(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, const double* A,
                          int64_t lda, const double* B, int64_t ldb, double tol, int* nm_out, emu_stream_t stream) {
  return bound_impl(h, layout, m, n, k, A, lda, B, ldb, tol, nm_out, stream, true);
}

}  // extern "C"

namespace {
// Shared by the Scheme I (p) and Scheme II (N moduli, norm scaling) auto
// entry points: selector class -> value, probe, escalation.
emu_status_t auto_impl(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, double alpha,
                       const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc,
                       double tol, int probe, int* p_used, emu_stream_t stream, bool scheme_II) {
  if (!h || !p_used || !A || !B || !C || m < 1 || n < 1 || k < 1 || !(tol > 0.0) || probe < 0 || !valid_layout(layout))
    return EMU_ERR_INVALID_ARG;
  if (!check_lds(layout, m, n, k, lda, ldb, ldc)) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  SelState* ss = sel_of(h);
  View v;
  normalize(layout, m, n, A, lda, B, ldb, &v);
  // device: features | histograms | probe indices | probe results [ref (hi,
  // lo) | sum |a||b|] | row and column maxima | digit sums; pinned host memory:
  // features, probabilities | probe results with the C entries
  const int pc = std::max(probe, 1);
  const size_t idx_bytes = (8 * static_cast<size_t>(pc) + 255) / 256 * 256;
  const size_t off_hist = 1024, off_idx = off_hist + feat_scratch(v), off_res = off_idx + idx_bytes;
  const size_t off_max = off_res + (24 * static_cast<size_t>(pc) + 255) / 256 * 256;
  const size_t max_bytes = (8 * static_cast<size_t>(v.M + v.N) + 15) / 16 * 16;
  const size_t zero_bytes = max_bytes + (scheme_II ? 0 : 4 * EMU_P_MAX * static_cast<size_t>(v.M + v.N) + 15) / 16 * 16;
  const size_t dev_need = off_max + zero_bytes;
  const size_t host_need = 1024 + 32 * static_cast<size_t>(pc);
  if (dev_need > ss->dev_bytes) {
    if (ss->dev) cudaFree(ss->dev);
    ss->dev = nullptr;
    ss->dev_bytes = 0;
    if (cudaMalloc(&ss->dev, dev_need) != cudaSuccess) {
      cudaGetLastError();
      return EMU_ERR_ALLOC;
    }
    // the decision's histograms start, and are left, at zero
    if (cudaMemset(ss->dev, 0, off_idx) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return EMU_ERR_CUDA;
    ss->dev_bytes = dev_need;
  }
  if (host_need > ss->host_bytes) {
    if (ss->host) cudaFreeHost(ss->host);
    ss->host = nullptr;
    ss->host_bytes = 0;
    if (cudaMallocHost(&ss->host, host_need) != cudaSuccess) {
      cudaGetLastError();
      return EMU_ERR_ALLOC;
    }
    ss->host_bytes = host_need;
  }
  if (!ss->side && (cudaStreamCreateWithFlags(&ss->side, cudaStreamNonBlocking) != cudaSuccess ||
                    cudaEventCreateWithFlags(&ss->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
                    cudaEventCreateWithFlags(&ss->ev_decide, cudaEventDisableTiming) != cudaSuccess ||
                    cudaEventCreateWithFlags(&ss->ev_probe, cudaEventDisableTiming) != cudaSuccess))
    return EMU_ERR_CUDA;
  auto* d_idx = reinterpret_cast<int32_t*>(ss->dev + off_idx);
  auto* d_ref = reinterpret_cast<double*>(ss->dev + off_res);
  auto* d_ab = d_ref + 2 * pc;
  auto* maxA = reinterpret_cast<unsigned long long*>(ss->dev + off_max);
  auto* maxB = maxA + v.M;
  auto* sums = reinterpret_cast<int32_t*>(ss->dev + off_max + max_bytes);  // digit sums of Scheme I's first attempt
  auto* h_dec = reinterpret_cast<float*>(ss->host);
  auto* h_res = reinterpret_cast<double*>(ss->host + 1024);
  const bool loaded = scheme_II ? ss->loaded_II : ss->loaded;
  // The decision (features and network, on sampled vectors), then the
  // exponent scan of the whole operands, which every attempt's product needs
  // whatever p it uses: the GPU scans while the host reads the decision and
  // enqueues the product.
  emu_status_t s = features_impl(v, k, tol, 64, reinterpret_cast<float*>(ss->dev), ss->dev + off_hist, st, true,
                                 loaded ? (scheme_II ? ss->params_II : ss->params) : nullptr, h_dec, reinterpret_cast<uint4*>(maxA),
                                 static_cast<int64_t>(zero_bytes / 16));
  if (s != EMU_OK) return s;
  if (cudaEventRecord(ss->ev_decide, st) != cudaSuccess) return EMU_ERR_CUDA;
  trace_begin(h, PH_SCAN, st);
  const cudaError_t es =
      launch_scan<double>(static_cast<const double*>(v.A), v.ldA, v.a_kcontig, v.M, maxA,
                          static_cast<const double*>(v.B), v.ldB, v.b_kcontig, v.N, maxB, k, 1, true, h->status, st);
  trace_end(h, PH_SCAN, st, 2);
  if (es != cudaSuccess) return cuda_err(es);
  // the probe's side stream starts after the caller's earlier work
  if (probe > 0 && (cudaEventRecord(ss->ev_fork, st) != cudaSuccess ||
                    cudaStreamWaitEvent(ss->side, ss->ev_fork, 0) != cudaSuccess))
    return EMU_ERR_CUDA;
  if (cudaEventSynchronize(ss->ev_decide) != cudaSuccess) return EMU_ERR_CUDA;
  const float* f = h_dec;
  const float* pr = f + 128;
  // value of class c and the largest value: p = 3 + c up to EMU_P_MAX, or
  // N = 6 + 2c up to EMU_NM_MAX
  const int top = scheme_II ? EMU_NM_MAX : EMU_P_MAX;
  const int step = scheme_II ? 2 : 1;
  const int base_v = scheme_II ? EMU_SEL_NM0 : EMU_SEL_P0;
  const int pb = scheme_II ? bound_nm_from_hist(f, k, tol) : bound_p_from_hist(f, k, tol);
  int p = pb;
  if (loaded) {  // smallest class whose cumulative predicted probability reaches 0.8
    float c = 0.f;
    int cls = kOut - 1;
    for (int o = 0; o < kOut; ++o) {
      c += pr[o];
      if (c >= 0.8f) {
        cls = o;
        break;
      }
    }
    // the top class is open-ended ("10 or more" / "20"): go to the largest value at once
    p = cls == kOut - 1 ? top : base_v + step * cls;
  }
  for (int attempt = 0; attempt < 3; ++attempt) {
    s = dgemm_scanned(h, layout, m, n, k, alpha, A, lda, B, ldb, C, ldc,
                      scheme_II ? EMU_SCHEME_II_NORM : EMU_SCHEME_I, p, maxA, maxB,
                      scheme_II || attempt > 0 ? nullptr : sums, stream);
    if (s != EMU_OK) return s;
    *p_used = p;
    if (probe == 0) return EMU_OK;
    if (attempt == 0) {
      // enqueued behind the product, so that its launches do not delay it
      probe_idx_kernel<<<1, 1, 0, ss->side>>>(
          0x9E3779B97F4A7C15ull ^ static_cast<uint64_t>(m * 1315423911u + n * 2654435761u + k), m, n, probe, d_idx);
      s = emu_probe_dd(h, layout, m, n, k, A, lda, B, ldb, probe, d_idx, d_ref, d_ab, ss->side);
      if (s != EMU_OK) return s;
      if (cudaEventRecord(ss->ev_probe, ss->side) != cudaSuccess) return EMU_ERR_CUDA;
    }
    if (attempt == 0 && cudaStreamWaitEvent(st, ss->ev_probe, 0) != cudaSuccess) return EMU_ERR_CUDA;
    judge_kernel<<<1, 256, 0, st>>>(C, ldc, layout != EMU_ROW_MAJOR, probe, d_idx, d_ref, d_ab, h_res);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return EMU_ERR_CUDA;
    const double* ref = h_res;
    const double* ab = ref + 2 * probe;
    const double* cv = ab + probe;
    double worst = 0.0;
    for (int q = 0; q < probe; ++q) {
      double d = std::fabs((cv[q] / alpha - ref[2 * q]) - ref[2 * q + 1]);
      double e = ab[q] > 0.0 ? d / ab[q] : (d > 0.0 ? INFINITY : 0.0);
      worst = std::max(worst, e);
    }
    if (worst <= tol) return EMU_OK;
    if (p >= top) return EMU_ERR_TOL_NOT_MET;
    // a miss at the top class goes straight to the largest value
    p = (attempt == 0 && p < base_v + step * (kOut - 1)) ? std::max(p + step, pb) : top;
    p = std::min(p, top);
  }
  return EMU_ERR_TOL_NOT_MET;
}
}  // namespace

extern "C" {

emu_status_t emu_dgemm_auto(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, double alpha,
                            const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc,
                            double tol, int probe, int* p_used, emu_stream_t stream) {
  return auto_impl(h, layout, m, n, k, alpha, A, lda, B, ldb, C, ldc, tol, probe, p_used, stream, false);
}

emu_status_t emu_dgemm_auto_II(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, double alpha,
                               const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc,
                               double tol, int probe, int* nm_used, emu_stream_t stream) {
  return auto_impl(h, layout, m, n, k, alpha, A, lda, B, ldb, C, ldc, tol, probe, nm_used, stream, true);
}



}  // extern "C"
