// api.cu -- the C ABI (include/emugemm.h): handle, workspace, host-side
// method constants, tensor maps, and the launch sequences of the hot path
// (scan -> split -> fused GEMM) for emu_dgemm / emu_sgemm / emu_zgemm and
// the exported intermediate steps.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "emu_internal.h"
#include "emu_handle.h"
#include "../../include/emugemm.h"

namespace emu {

// ================================================================ constants
// Greedy descending list of pairwise-coprime integers from 256 (Sec. II-C-2
// names 256, 255, 253, ...).
int host_moduli(int nm, int32_t* out) {
  int cnt = 0;
  for (int x = 256; x >= 2 && cnt < nm; --x) {
    bool ok = true;
    for (int j = 0; j < cnt && ok; ++j) {
      int a = x, b = out[j];
      while (b) {
        int t = a % b;
        a = b;
        b = t;
      }
      ok = (a == 1);
    }
    if (ok) out[cnt++] = x;
  }
  return cnt;
}

// K_c: largest multiple of 256 such that every triangular partial C_s of
// Eq. (2) stays within int32 for the slice ranges (leading slice in
// [-128, 127], tails in [0, 255]), from interval products per pair.
int64_t host_chunk_len_I(int p) {
  int64_t worst = 0;
  for (int s = 0; s < p; ++s) {
    int64_t hi = 0, lo = 0;
    for (int i = 0; i <= s; ++i) {
      int64_t alo = i == 0 ? -128 : 0, ahi = i == 0 ? 127 : 255;
      int64_t blo = (s - i) == 0 ? -128 : 0, bhi = (s - i) == 0 ? 127 : 255;
      int64_t c[4] = {alo * blo, alo * bhi, ahi * blo, ahi * bhi};
      int64_t mx = c[0], mn = c[0];
      for (int q = 1; q < 4; ++q) {
        mx = c[q] > mx ? c[q] : mx;
        mn = c[q] < mn ? c[q] : mn;
      }
      hi += mx;
      lo += mn;
    }
    worst = hi > worst ? hi : worst;
    worst = -lo > worst ? -lo : worst;
  }
  int64_t lim = 2147483647LL / worst;
  return lim - lim % 256;
}

// K_c for the E4M3 engine: every |d_i d_j| <= 16 * 16, so C_s grows by at
// most (s+1) * 256 per unit of K; largest multiple of 256 keeping every FP32
// partial sum within 2^24 (where FP32 holds all integers exactly).
int64_t host_chunk_len_F8(int p) {
  int64_t worst = 0;
  for (int s = 0; s < p; ++s) worst = std::max<int64_t>(worst, static_cast<int64_t>(s + 1) * 16 * 16);
  int64_t lim = (int64_t{1} << 24) / worst;
  return lim - lim % 256;
}

namespace {
// little-endian 32-bit limb integers
using Limbs = std::vector<uint32_t>;
void limbs_mul_small(Limbs& a, uint32_t v) {
  uint64_t c = 0;
  for (auto& w : a) {
    c += static_cast<uint64_t>(w) * v;
    w = static_cast<uint32_t>(c);
    c >>= 32;
  }
  if (c) a.push_back(static_cast<uint32_t>(c));
}
uint32_t limbs_mod_small(const Limbs& a, uint32_t m) {
  uint64_t r = 0;
  for (size_t i = a.size(); i-- > 0;) r = ((r << 32) | a[i]) % m;
  return static_cast<uint32_t>(r);
}
int limbs_bitlen(const Limbs& a) {
  for (size_t i = a.size(); i-- > 0;)
    if (a[i]) {
      int b = 32;
      while (!((a[i] >> (b - 1)) & 1u)) --b;
      return static_cast<int>(32 * i) + b;
    }
  return 0;
}
Limbs limbs_P(int nm) {
  int32_t mods[kMaxModuli + 4];
  host_moduli(nm, mods);
  Limbs P{1u};
  for (int l = 0; l < nm; ++l) limbs_mul_small(P, static_cast<uint32_t>(mods[l]));
  return P;
}
// modular inverse by the extended Euclidean algorithm
int64_t inv_mod(int64_t a, int64_t m) {
  int64_t g = m, x = 0, x1 = 1, a1 = a % m;
  while (a1) {
    int64_t q = g / a1;
    int64_t t = g - q * a1;
    g = a1;
    a1 = t;
    t = x - q * x1;
    x = x1;
    x1 = t;
  }
  return ((x % m) + m) % m;
}
}  // namespace

// b = floor((floor(log2 P) - 1 - ceil(log2 k)) / 2); complex uses -2.
int host_scale_bits_II(int nm, int64_t k, int is_complex) {
  int lp = limbs_bitlen(limbs_P(nm)) - 1;
  int c = 0;
  while ((int64_t{1} << c) < k) ++c;
  int num = lp - (is_complex ? 2 : 1) - c;
  return num >= 0 ? num / 2 : -((-num + 1) / 2);
}

// Norm-based scaling: one exponent h for both operands (the product stays
// symmetric in A and B, whichever one is stored transposed), 2h + 1 <=
// floor(log2 P).
void host_norm_halves_II(int nm, int* hA, int* hB) {
  const int L = limbs_bitlen(limbs_P(nm)) - 2;  // floor(log2 P) - 1
  *hA = L >= 0 ? L / 2 : -((-L + 1) / 2);
  *hB = *hA;
}

void host_mod_tables(int nm, ModTables* t) {
  std::memset(t, 0, sizeof(*t));
  int32_t mods[kMaxModuli];
  host_moduli(nm, mods);
  for (int l = 0; l < nm; ++l) {
    const int32_t m = mods[l], hi = (m - 1) / 2;
    t->mods[l] = static_cast<uint32_t>(m);
    t->off[l] = m - 1 - hi;
    t->inv[l] = 1.0f / static_cast<float>(m);
    t->offinv[l] = static_cast<float>(t->off[l]) / static_cast<float>(m);
    t->offhinv[l] = static_cast<float>(t->off[l] + 0.5) / static_cast<float>(m);
    int64_t v = 1 % m;  // 2^(16 j) mod m
    for (int j = 0; j < kResDigits; ++j) {
      t->pow16[l][j] = static_cast<int32_t>(v > hi ? v - m : v);
      v = (v << 16) % m;
    }
    t->mf[l] = static_cast<float>(m);
    t->offf[l] = static_cast<float>(t->off[l]);
    v = 1 % m;  // 2^(14 j) mod m
    for (int j = 0; j < kResDigitsF; ++j) {
      t->pow14f[l][j] = static_cast<float>(v > hi ? v - m : v);
      v = (v << 14) % m;
    }
  }
}

void host_crt_tables(int nm, CrtTables* t) {
  std::memset(t, 0, sizeof(*t));
  int32_t mods[kMaxModuli];
  host_moduli(nm, mods);
  t->nm = nm;
  Limbs P = limbs_P(nm);
  for (int i = 0; i < kCrtLimbs && i < static_cast<int>(P.size()); ++i) t->P[i] = P[i];
  // floor(P/2)
  for (int i = 0; i < kCrtLimbs; ++i)
    t->Phalf[i] = (t->P[i] >> 1) | (i + 1 < kCrtLimbs ? (t->P[i + 1] << 31) : 0u);
  double pd = 0.0;
  for (int i = kCrtLimbs - 1; i >= 0; --i) pd = pd * 4294967296.0 + t->P[i];
  t->invP = 1.0 / pd;
  for (int l = 0; l < nm; ++l) {
    Limbs Pl{1u};
    for (int j = 0; j < nm; ++j)
      if (j != l) limbs_mul_small(Pl, static_cast<uint32_t>(mods[j]));
    uint32_t pm = limbs_mod_small(Pl, static_cast<uint32_t>(mods[l]));
    int64_t q = inv_mod(pm, mods[l]);
    limbs_mul_small(Pl, static_cast<uint32_t>(q));
    for (int i = 0; i < kCrtLimbs && i < static_cast<int>(Pl.size()); ++i) t->w[l][i] = Pl[i];
  }
}

void host_crt_pair_tables(int nm, CrtPairTables* t) {
  std::memset(t, 0, sizeof(*t));
  int32_t mods[kMaxModuli];
  host_moduli(nm, mods);
  t->nm = nm;
  const Limbs P = limbs_P(nm);
  const int bl = limbs_bitlen(P);
  for (size_t i = 0; i < P.size() && i < kCrtLimbs; ++i) t->P[i] = P[i];
  for (int i = 0; i < kCrtLimbs; ++i) t->Phalf[i] = (t->P[i] >> 1) | (i + 1 < kCrtLimbs ? (t->P[i + 1] << 31) : 0u);
  t->limbs = std::max(2, (bl + 31) / 32);
  const int e = std::max(0, bl - 32);
  t->sh = e - 32 * (t->limbs - 2);
  if (e == 0) t->sh = 0;
  t->frac = bl - 1 - e;
  {  // floor(2^(63 + bl) / P) by binary long division (64 quotient bits; P a power of two: all ones)
    Limbs rem(P.size() + 1, 0u);
    auto ge = [&] {
      if (rem[P.size()]) return true;
      for (size_t i = P.size(); i-- > 0;)
        if (rem[i] != P[i]) return rem[i] > P[i];
      return true;
    };
    uint64_t q = 0;
    bool over = false;
    for (int b = 63 + bl; b >= 0; --b) {
      uint32_t carry = b == 63 + bl ? 1u : 0u;
      for (auto& w : rem) {
        const uint32_t top = w >> 31;
        w = (w << 1) | carry;
        carry = top;
      }
      over = over || (q >> 63) != 0;
      q <<= 1;
      if (ge()) {
        uint64_t br = 0;
        for (size_t i = 0; i < rem.size(); ++i) {
          const uint64_t d = static_cast<uint64_t>(rem[i]) - (i < P.size() ? P[i] : 0u) - br;
          rem[i] = static_cast<uint32_t>(d);
          br = d >> 63;
        }
        q |= 1u;
      }
    }
    t->recip = over ? ~uint64_t{0} : q;
  }
  for (int i = 0; 2 * i < nm; ++i) {
    const int64_t m = mods[2 * i], m2 = 2 * i + 1 < nm ? mods[2 * i + 1] : 1, mm = m * m2;
    const int64_t lo = m2 * inv_mod(m2 % m, m) % mm, hi = m2 > 1 ? m * inv_mod(m % m2, m2) % mm : 0;
    t->c[i] = static_cast<uint32_t>(lo) | (static_cast<uint32_t>(hi) << 16);
    t->off[i] = static_cast<uint32_t>(((int64_t{1} << 25) / mm + 1) * mm);
    Limbs W{1u};
    for (int j = 0; j < nm; ++j)
      if (j / 2 != i) limbs_mul_small(W, static_cast<uint32_t>(mods[j]));
    limbs_mul_small(W, static_cast<uint32_t>(inv_mod(limbs_mod_small(W, static_cast<uint32_t>(mm)), mm)));
    for (size_t j = 0; j < W.size() && j < kCrtLimbs; ++j) t->w[i][j] = W[j];
  }
}

const MethodTables& method_tables(int nm) {
  static MethodTables tabs[kMaxModuli + 1];
  static std::once_flag once[kMaxModuli + 1];
  std::call_once(once[nm], [nm] {
    host_mod_tables(nm, &tabs[nm].mod);
    host_crt_tables(nm, &tabs[nm].crt);
    host_crt_pair_tables(nm, &tabs[nm].pair);
  });
  return tabs[nm];
}

// ================================================================ tensor maps
namespace {
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                              CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                              CUtensorMapFloatOOBfill);
EncodeFn get_encode() {
  static EncodeFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(p);
  });
  return fn;
}
}  // namespace

bool make_tmap_i8(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows, uint32_t box_rows,
                  uint32_t box_bytes) {
  EncodeFn enc = get_encode();
  if (!enc) return false;
  if (box_bytes != 32 && box_bytes != 128) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols};
  cuuint32_t box[2] = {box_bytes, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   box_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_32B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// ================================================================ misc kernels
template <typename T>
__global__ void scale_c_kernel(T* C, int64_t ldc, int64_t m, int64_t n, double beta) {
  int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= m * n) return;
  int64_t i = idx / n, j = idx % n;
  T* p = C + i * ldc + j;
  *p = beta == 0.0 ? T(0) : static_cast<T>(__dmul_rn(beta, static_cast<double>(*p)));
}
// k == 0: C = beta * C for complex beta (C not read when beta == 0); float
// C (CGEMM) is widened, updated in binary64 and rounded once per part.
template <typename T>
__global__ void scale_z_kernel(T* C, int64_t ldc, int64_t m, int64_t n, double br, double bi) {
  int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= m * n) return;
  int64_t i = idx / n, j = idx % n;
  T* p = C + 2 * (i * ldc + j);
  if (br == 0.0 && bi == 0.0) {
    p[0] = T(0);
    p[1] = T(0);
    return;
  }
  double cr = static_cast<double>(p[0]), ci = static_cast<double>(p[1]);
  p[0] = static_cast<T>(__fma_rn(br, cr, -__dmul_rn(bi, ci)));
  p[1] = static_cast<T>(__fma_rn(br, ci, __dmul_rn(bi, cr)));
}

// One warp waits on an mbarrier that nothing arrives on; the bounded wait
// gives up after `limit` cycles and records the timeout.
__global__ void selftest_wait_kernel(int* status, long long limit) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncwarp();
  if (threadIdx.x == 0 && !mbar_wait_bounded(&bar, 0, limit)) set_status(status, ST_TIMEOUT);
}

}  // namespace emu

using namespace emu;

// ================================================================ handle
// What was behind this thread's last EMU_ERR_CUDA (emu_last_cuda_error).
static thread_local const char* g_last_cuda_error = "no error";
emu_status_t emu::cuda_err(cudaError_t e) {
  if (e == cudaSuccess) return EMU_OK;
  g_last_cuda_error = cudaGetErrorString(e);
  cudaGetLastError();  // reported here: not left for the thread's next query
  return EMU_ERR_CUDA;
}
static emu_status_t tmap_err() {
  g_last_cuda_error = "tensor map encoding failed";
  return EMU_ERR_CUDA;
}

namespace emu {
// EMU_FAULT: host-side fault injection (read once).  alloc: every
// library-owned workspace allocation fails, alloc:N every one of more than N
// bytes; launch: the fused GEMM launch of every product, zero, scan, norm or
// split: every launch of that step before it.  A launch fails as a launch would
// (cudaErrorLaunchFailure); nothing runs on the device that could fault.
static int fault_mode() {
  static int v = -1;
  if (v < 0) {
    static const char* const names[] = {"", "alloc", "launch", "zero", "scan", "norm", "split"};
    const char* e = std::getenv("EMU_FAULT");
    int x = 0;
    for (int i = FAULT_ALLOC; e && i <= FAULT_SPLIT; ++i)
      if (std::strcmp(e, names[i]) == 0) x = i;
    if (e && std::strncmp(e, "alloc:", 6) == 0) x = FAULT_ALLOC;
    v = x;
  }
  return v;
}
static bool fault_alloc(size_t bytes) {
  static const size_t most = [] {
    const char* e = std::getenv("EMU_FAULT");
    return e && std::strncmp(e, "alloc:", 6) == 0 ? static_cast<size_t>(std::strtoull(e + 6, nullptr, 10)) : 0;
  }();
  return fault_mode() == FAULT_ALLOC && bytes > most;
}
cudaError_t fault_step(FaultStep step) { return fault_mode() == step ? cudaErrorLaunchFailure : cudaSuccess; }
static cudaError_t fault_launch() { return fault_step(FAULT_GEMM); }

namespace {
struct StreamMem {
  cudaStream_t st;
  bool capturing() const {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) == cudaSuccess) return cs != cudaStreamCaptureStatusNone;
    cudaGetLastError();
    return true;
  }
  void* alloc(size_t n) const {
    void* p = nullptr;
    if (fault_alloc(n)) return nullptr;
    if (cudaMallocAsync(&p, n, st) == cudaSuccess) return p;
    cudaGetLastError();
    return nullptr;
  }
  void release(void* p) const { cudaFreeAsync(p, st); }
};
struct SyncMem {  // after a device synchronisation
  void release(void* p) const { cudaFree(p); }
};
}  // namespace

emu_status_t handle_workspace(emu_handle_s* h, size_t bytes, cudaStream_t st, uint8_t** out, bool optional) {
  if (h->ws_user) {
    if (bytes > h->ws_user_bytes) return EMU_ERR_ALLOC;
    *out = static_cast<uint8_t*>(h->ws_user);
    return EMU_OK;
  }
  StreamMem mem{st};
  return ws_reserve(h->ws, bytes, optional, mem, out) ? EMU_OK : EMU_ERR_ALLOC;
}
}  // namespace emu

extern "C" {

emu_status_t emu_create(emu_handle_t* out, int device) {
  if (!out) return EMU_ERR_INVALID_ARG;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
    cudaGetLastError();
    return EMU_ERR_CUDA;
  }
  if (cudaSetDevice(device) != cudaSuccess) return EMU_ERR_CUDA;
  emu_handle_s* h = new (std::nothrow) emu_handle_s();
  if (!h) return EMU_ERR_ALLOC;
  h->device = device;
  cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, device);
  if (cudaMalloc(&h->status, sizeof(int)) != cudaSuccess) {
    delete h;
    return EMU_ERR_ALLOC;
  }
  cudaMemset(h->status, 0, sizeof(int));
  if (cudaDeviceSynchronize() != cudaSuccess) {
    cudaFree(h->status);
    delete h;
    return EMU_ERR_CUDA;
  }
  *out = h;
  return EMU_OK;
}

emu_status_t emu_destroy(emu_handle_t h) {
  if (!h) return EMU_OK;
  cudaSetDevice(h->device);
  cudaDeviceSynchronize();
  handle_release_extras(h);
  SyncMem mem;
  ws_close(h->ws, mem);
  if (h->status) cudaFree(h->status);
  delete h;
  return EMU_OK;
}

emu_status_t emu_get_status(emu_handle_t h, emu_stream_t stream) {
  if (!h) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (cudaStreamSynchronize(st) != cudaSuccess) return EMU_ERR_CUDA;
  int v = 0;
  if (cudaMemcpy(&v, h->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return EMU_ERR_CUDA;
  cudaMemset(h->status, 0, sizeof(int));
  cudaDeviceSynchronize();
  if (v & ST_TIMEOUT) return EMU_ERR_TIMEOUT;
  if (v & ST_NONFINITE) return EMU_ERR_NONFINITE;
  return EMU_OK;
}

emu_status_t emu_selftest_wait(emu_handle_t h, int64_t limit_cycles, emu_stream_t stream) {
  if (!h) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  long long lim = limit_cycles < 1000 ? 1000 : (limit_cycles > 2000000000LL ? 2000000000LL : limit_cycles);
  selftest_wait_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(h->status, lim);
  return cuda_err(cudaGetLastError());
}

const char* emu_last_cuda_error(void) { return g_last_cuda_error; }

const char* emu_status_string(emu_status_t s) {
  switch (s) {
    case EMU_OK: return "EMU_OK";
    case EMU_ERR_INVALID_ARG: return "EMU_ERR_INVALID_ARG";
    case EMU_ERR_UNSUPPORTED: return "EMU_ERR_UNSUPPORTED";
    case EMU_ERR_NONFINITE: return "EMU_ERR_NONFINITE";
    case EMU_ERR_CUDA: return "EMU_ERR_CUDA";
    case EMU_ERR_ALLOC: return "EMU_ERR_ALLOC";
    case EMU_ERR_TIMEOUT: return "EMU_ERR_TIMEOUT";
    case EMU_ERR_TOL_NOT_MET: return "EMU_ERR_TOL_NOT_MET";
  }
  return "EMU_ERR_UNKNOWN";
}

int64_t emu_split_rows(int64_t rows) { return split_rows(rows); }
int64_t emu_split_cols_I(int64_t k, int p) { return split_cols_I(k, p); }
int64_t emu_split_cols_II(int64_t k) { return split_cols_II(k); }
int64_t emu_chunk_len_I(int p) { return p >= 1 ? host_chunk_len_I(p) : 0; }
int64_t emu_chunk_len_F8(int p) { return p >= 1 ? host_chunk_len_F8(p) : 0; }
int emu_moduli(int nm, int32_t* mods) { return mods ? host_moduli(nm, mods) : 0; }
int emu_scale_bits_II(int nm, int64_t k, int is_complex) { return host_scale_bits_II(nm, k, is_complex); }

emu_status_t emu_set_workspace(emu_handle_t h, void* ws, size_t bytes) {
  if (!h) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  if (h->ws.p) {
    cudaDeviceSynchronize();
    SyncMem mem;
    if (!ws_drop(h->ws, mem)) return EMU_ERR_ALLOC;
  }
  h->ws_user = ws;
  h->ws_user_bytes = ws ? bytes : 0;
  if (ws && (reinterpret_cast<uintptr_t>(ws) & 255u)) return EMU_ERR_INVALID_ARG;
  return EMU_OK;
}

}  // extern "C"

// ================================================================ planning
namespace emu {

static inline size_t al256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

// EMU_F8_ENGINE=mma selects the warp-level FP8 kernel for E4M3 slices (for
// comparison); the default is the tcgen05 kernel.
static bool f8_engine_mma() {
  static int v = -1;
  if (v < 0) {
    const char* e = std::getenv("EMU_F8_ENGINE");
    v = (e && std::strcmp(e, "mma") == 0) ? 1 : 0;
  }
  return v == 1;
}

// EMU_II_ENGINE=mma selects the INT8 mma.sync kernel for Scheme II (for
// comparison; identical results); the default is the bf16 tcgen05 kernel.
bool ii_engine_tc() {
  static int v = -1;
  if (v < 0) {
    const char* e = std::getenv("EMU_II_ENGINE");
    v = (e && std::strcmp(e, "mma") == 0) ? 0 : 1;
  }
  return v == 1;
}

Plan plan_I(int64_t m, int64_t n, int64_t k, int p) {
  Plan pl{};
  pl.rows_a = split_rows(m);
  pl.rows_b = split_rows(n);
  pl.cols = split_cols_I(k, p);
  size_t off = 0;
  pl.off_maxA = off; off += al256(8 * static_cast<size_t>(m > 0 ? m : 1));
  pl.off_maxB = off; off += al256(8 * static_cast<size_t>(n > 0 ? n : 1));
  pl.off_EA = off; off += al256(4 * static_cast<size_t>(m > 0 ? m : 1));
  pl.off_FB = off; off += al256(4 * static_cast<size_t>(n > 0 ? n : 1));
  pl.off_hatA = off; off += al256(static_cast<size_t>(pl.rows_a) * pl.cols);
  pl.off_hatB = off; off += al256(static_cast<size_t>(pl.rows_b) * pl.cols);
  pl.bytes = off;
  return pl;
}

// EMU_I_ENGINE=mma selects the INT8 mma.sync kernel for Scheme I (for
// comparison; identical results); the default is the bf16 tcgen05 path.
static bool i_engine_tc() {
  static int v = -1;
  if (v < 0) {
    const char* e = std::getenv("EMU_I_ENGINE");
    v = (e && std::strcmp(e, "mma") == 0) ? 0 : 1;
  }
  return v == 1;
}

PlanTri plan_tri(int64_t rows, int64_t n, int64_t k, int p) {
  const TriLayout L = tri_layout(rows, n, k, p);
  PlanTri pl{};
  size_t off = 0;
  pl.off_maxA = off; off += al256(8 * static_cast<size_t>(rows));
  pl.off_maxB = off; off += al256(8 * static_cast<size_t>(n));
  pl.off_sumA = off; off += al256(4 * static_cast<size_t>(p) * rows);
  pl.off_sumB = off; off += al256(4 * static_cast<size_t>(p) * n);
  pl.zero_bytes = off;
  pl.off_EA = off; off += al256(4 * static_cast<size_t>(rows));
  pl.off_FB = off; off += al256(4 * static_cast<size_t>(n));
  const size_t vec = 2 * static_cast<size_t>(tri_num_planes(p)) * static_cast<size_t>(L.kpad);
  pl.off_planesA = off; off += al256(vec * static_cast<size_t>(rows));
  pl.off_planesB = off; off += al256(vec * static_cast<size_t>(n));
  pl.off_Cs = off; off += al256(L.Cs_bytes);
  pl.bytes = off;
  return pl;
}

// A pass holds A's digit planes and the int32 output planes of at most this
// many bytes (about 8000 rows at n = k = 8192, p = 8); larger products run
// in row passes, so that a handle's workspace grows with B's planes alone.
constexpr int64_t kTriPassBytes = int64_t{8} << 30;
// K beyond this keeps the INT8 kernel: the int32 digit sums (|d| <= 128 per
// element) and the number of K chunks stay small below it.
constexpr int64_t kTriMaxK = int64_t{1} << 20;

// More than eight slices (FP64 accuracy needs eight; the rest serves wide
// exponent ranges) take this path only from 2^33 multiply-adds.  This line is
// not where it stops paying: it is faster below as well (n = 1344, p = 12: 0.41
// ms against 2.61).  But then the largest p costs little more than a chosen one
// plus the choice, whose waits for the device are 30 to 50 us of a call of 220
// to 350, and emu_dgemm_auto is to gain 1.05x over the fixed largest p at n =
// 1024 .. 1536: it does by 1.47x with this line, by 1.02-1.03x without (1.04-1.06
// with the probe's sums enqueued before the product instead of behind it).  It
// can go when the automatic call costs some 20 us less.
constexpr int kTriSmallP = 8;
constexpr int64_t kTriLargeWork = int64_t{1} << 33;

bool tri_can(int64_t m, int64_t n, int64_t k, int p) {
  if (!i_engine_tc() || k < 1 || k > kTriMaxK) return false;
  // plane rows are TMA coordinates (int32)
  return (m > n ? m : n) <= INT32_MAX / tri_num_planes(p) / 2;
}

// Long and narrow products of short K: what counts is not the products but
// the bf16 planes (46 bytes per operand element at p = 8, the INT8 slices 8)
// and the int32 planes of 32 columns at least, written and read again.  From
// 20 items per SM on (smaller products are bound by their launches) INT8
// mma.sync against bf16 planes, us, 262144 rows:
//   p = 8: 8 columns, K = 32 383 / 659, 64 512 / 663, 128 771 / 807, 256 1383
//          / 1340; 32 columns, K = 64 580 / 702, 128 829 / 843; 64 columns,
//          K = 32 709 / 872, 64 958 / 872; 128 columns, K = 32 1218 / 1255
//   p = 4: 8 columns, K = 64 292 / 380, 128 367 / 414; 32 columns, K = 64 369 /
//          399, 128 452 / 430; 64 columns, K = 32 491 / 496
//   p = 3: 8 columns, K = 64 258 / 282, 128 312 / 312; 16 columns, K = 64 309 / 285
//   p = 2: 8 columns, K = 32 219 / 231, 64 233 / 231
// and short and wide: p = 8, 8 x 262144, K = 32 464 / 542, 64 722 / 563; 32 x
// 262144, K = 32 542 / 585; p = 6, 8 x 262144, K = 32 370 / 429; p = 4 292 / 312.
static bool tri_pays(int64_t m, int64_t n, int64_t k, int p) {
  if (p > kTriSmallP && static_cast<double>(m) * static_cast<double>(n) * static_cast<double>(k) < kTriLargeWork)
    return false;
  if (p < 3 || (m + tri_tile_m() - 1) / tri_tile_m() * ((n + tri_tile_n() - 1) / tri_tile_n()) * tri_num_units(p) <
                   20 * 152)
    return true;
  const int64_t k32 = (k + 31) / 32 * 32;
  if (n <= 64 && k32 * std::max<int64_t>(n, 16) <= 2048 && (p > 3 || n <= 8)) return false;
  return !(p >= 6 && m <= 8 && k <= 32);
}

int64_t tri_rows(int64_t m, int64_t n, int64_t k, int p) {
  if (!tri_can(m, n, k, p) || !tri_pays(m, n, k, p)) return 0;
  auto pass = [&](int64_t rows) {
    const TriLayout L = tri_layout(rows, n, k, p);
    return static_cast<int64_t>(L.Cs_bytes) + 2 * static_cast<int64_t>(tri_num_planes(p)) * rows * L.kpad;
  };
  int64_t rows = m;
  while (pass(rows) > kTriPassBytes && rows > tri_tile_m())
    rows = ((rows + 1) / 2 + tri_tile_m() - 1) / tri_tile_m() * tri_tile_m();
  return pass(rows) > 4 * kTriPassBytes ? 0 : rows;  // extremely wide or deep: the INT8 kernel
}

size_t workspace_I(int64_t m, int64_t n, int64_t k, int p, bool f8) {
  // emu_workspace_size does not know the layout, and a column-major product
  // runs transposed: room for either
  size_t bytes = std::max(plan_I(m, n, k, p).bytes, plan_I(n, m, k, p).bytes);
  if (f8 || m < 1 || n < 1) return bytes;
  for (int t = 0; t < 2; ++t) {
    const int64_t M = t ? n : m, N = t ? m : n, rows = tri_rows(M, N, k, p);
    if (rows > 0) bytes = std::max(bytes, plan_tri(rows, N, k, p).bytes);
  }
  return bytes;
}

// es: bytes per residue (1: INT8 planes, 2: bf16 planes of the tcgen05 kernel)
Plan plan_II(int64_t m, int64_t n, int64_t k, int nm, int nsets, int es) {
  Plan pl{};
  pl.rows_a = split_rows(m);
  pl.rows_b = split_rows(n);
  pl.cols = split_cols_II(k);
  size_t off = 0;
  pl.off_maxA = off; off += al256(8 * static_cast<size_t>(m > 0 ? m : 1));
  pl.off_maxB = off; off += al256(8 * static_cast<size_t>(n > 0 ? n : 1));
  // norm-based scaling: 128-bit sums of squares, zeroed with the maxima
  pl.off_accA = off; off += al256(16 * static_cast<size_t>(m > 0 ? m : 1));
  pl.off_accB = off; off += al256(16 * static_cast<size_t>(n > 0 ? n : 1));
  pl.off_EA = off; off += al256(4 * static_cast<size_t>(m > 0 ? m : 1));
  pl.off_FB = off; off += al256(4 * static_cast<size_t>(n > 0 ? n : 1));
  pl.off_hatA = off; off += al256(static_cast<size_t>(es) * nsets * nm * pl.rows_a * pl.cols);
  pl.off_hatB = off; off += al256(static_cast<size_t>(es) * nsets * nm * pl.rows_b * pl.cols);
  // tcgen05 kernel: the residue planes (one byte per output and modulus; row
  // tiles rounded to whole CTA-pair tiles)
  pl.off_scratch = off; off += es == 2 ? al256(gemm_II_tc_residue_bytes(m, n, nm, nsets == 3, 2)) : 0;
  pl.bytes = off;
  return pl;
}

// Row-major view of the product: C (M x N) = Aop (M x K) * Bop (K x N) where
// Aop's rows are reduction vectors read with (ldA, a_kcontig) and Bop's
// columns with (ldB, b_kcontig).  Column-major calls are mapped onto the
// transposed row-major product C^T = B^T A^T.
void normalize(emu_layout_t layout, int64_t m, int64_t n, const void* A, int64_t lda, const void* B,
               int64_t ldb, View* v) {
  if (layout == EMU_ROW_MAJOR) {
    v->M = m;
    v->N = n;
    v->A = A;
    v->ldA = lda;
    v->a_kcontig = true;
    v->B = B;
    v->ldB = ldb;
    v->b_kcontig = false;
  } else {
    v->M = n;
    v->N = m;
    v->A = B;
    v->ldA = ldb;
    v->a_kcontig = true;
    v->B = A;
    v->ldB = lda;
    v->b_kcontig = false;
  }
}

bool check_lds(emu_layout_t layout, int64_t m, int64_t n, int64_t k, int64_t lda, int64_t ldb,
               int64_t ldc) {
  if (layout == EMU_ROW_MAJOR)
    return lda >= (k > 1 ? k : 1) && ldb >= (n > 1 ? n : 1) && ldc >= (n > 1 ? n : 1);
  return lda >= (m > 1 ? m : 1) && ldb >= (k > 1 ? k : 1) && ldc >= (m > 1 ? m : 1);
}

template <typename T>
emu_status_t run_tri(emu_handle_s* h, const View& v, int64_t k, int p, double alpha, double beta, void* C,
                     int64_t ldc, int out_mode, cudaStream_t st, uint8_t* ws, int64_t rows, int phase) {
  const PlanTri pl = plan_tri(rows, v.N, k, p);
  auto* maxA = reinterpret_cast<unsigned long long*>(ws + pl.off_maxA);
  auto* maxB = reinterpret_cast<unsigned long long*>(ws + pl.off_maxB);
  auto* sumA = reinterpret_cast<int32_t*>(ws + pl.off_sumA);
  auto* sumB = reinterpret_cast<int32_t*>(ws + pl.off_sumB);
  auto* EA = reinterpret_cast<int32_t*>(ws + pl.off_EA);
  auto* FB = reinterpret_cast<int32_t*>(ws + pl.off_FB);
  auto* planesA = reinterpret_cast<uint16_t*>(ws + pl.off_planesA);
  auto* planesB = reinterpret_cast<uint16_t*>(ws + pl.off_planesB);
  const T* A = static_cast<const T*>(v.A);
  const T* B = static_cast<const T*>(v.B);
  // maxima and digit sums start at zero; in a first pass over A with B one
  // memset and one scan serve both operands
  const bool both = phase == 0;
  cudaError_t e = cudaSuccess;
  if (phase != 2) {
    trace_begin(h, PH_SCAN, st);
    if (both) {
      if (v.sums && rows >= v.M) {  // zeroed by the caller
        sumA = v.sums;
        sumB = v.sums + static_cast<int64_t>(p) * v.M;
      } else {
        e = launch_zero(ws, pl.zero_bytes, st);
      }
      if (e == cudaSuccess && !v.maxA)
        e = launch_scan<T>(A, v.ldA, v.a_kcontig, std::min(rows, v.M), maxA, B, v.ldB, v.b_kcontig, v.N, maxB, k, 1,
                           true, h->status, st);
    } else {
      e = cudaMemsetAsync(sumB, 0, sizeof(*sumB) * p * v.N, st);
      if (e == cudaSuccess && !v.maxB) e = launch_scan_one<T>(B, v.ldB, v.b_kcontig, v.N, k, 1, maxB, h->status, st);
    }
    trace_end(h, PH_SCAN, st, both ? 2 : 1);
    if (e != cudaSuccess) return cuda_err(e);
    trace_begin(h, PH_SPLIT, st);
    e = launch_split_tri<T>(B, v.ldB, v.b_kcontig, v.N, k, p, v.maxB ? v.maxB : maxB, planesB, FB, sumB, h->num_sms,
                            st);
    trace_end(h, PH_SPLIT, st, 1);
    if (e != cudaSuccess) return cuda_err(e);
  }
  if (phase == 1) return EMU_OK;
  const int np = tri_num_planes(p);
  for (int64_t r0 = 0; r0 < v.M; r0 += rows) {
    const int64_t m = std::min(rows, v.M - r0);
    const T* Ar = A + (v.a_kcontig ? r0 * v.ldA : r0);
    if (!both || r0 > 0) {
      trace_begin(h, PH_SCAN, st);
      e = cudaMemsetAsync(sumA, 0, sizeof(*sumA) * p * m, st);
      if (e == cudaSuccess && !v.maxA) e = launch_scan_one<T>(Ar, v.ldA, v.a_kcontig, m, k, 1, maxA, h->status, st);
      trace_end(h, PH_SCAN, st, 1);
      if (e != cudaSuccess) return cuda_err(e);
    }
    trace_begin(h, PH_SPLIT, st);
    e = launch_split_tri<T>(Ar, v.ldA, v.a_kcontig, m, k, p, v.maxA ? v.maxA + r0 : maxA, planesA, EA, sumA,
                            h->num_sms, st);
    trace_end(h, PH_SPLIT, st, 1);
    if (e != cudaSuccess) return cuda_err(e);
    GemmTriArgs a{};
    a.L = tri_layout(rows, v.N, k, p);  // the workspace's layout, for fewer rows in the last pass
    a.L.tiles_m = (m + tri_tile_m() - 1) / tri_tile_m();
    const uint64_t row_bytes = 2 * static_cast<uint64_t>(a.L.kpad);
    // boxes no higher than the product (in steps of the 8-row swizzle atoms
    // and of the 32 columns that the MMAs compute)
    const auto box_a = static_cast<uint32_t>(std::min<int64_t>((m + 7) / 8 * 8, tri_tile_m()));
    const auto box_b = static_cast<uint32_t>(std::min<int64_t>((v.N + 31) / 32 * 32, tri_tile_n()));
    CUtensorMap ta, tb;
    if (!make_tmap_i8(&ta, planesA, row_bytes, static_cast<uint64_t>(m) * np, box_a, 128) ||
        !make_tmap_i8(&tb, planesB, row_bytes, static_cast<uint64_t>(v.N) * np, box_b, 128))
      return tmap_err();
    a.descA = &ta;
    a.descB = &tb;
    a.box_bytes = static_cast<int>((box_a + box_b) * 128);
    a.M = static_cast<int>(m);
    a.N = static_cast<int>(v.N);
    a.K = k;
    a.Cs = reinterpret_cast<int32_t*>(ws + pl.off_Cs);
    a.sumA = sumA;
    a.sumB = sumB;
    a.EA = EA;
    a.FB = FB;
    a.alpha = alpha;
    a.beta = beta;
    a.C = static_cast<uint8_t*>(C) + (out_mode == OUT_F32 ? 4 : 8) * r0 * ldc;
    a.ldc = ldc;
    a.status = h->status;
    a.num_sms = h->num_sms;
    trace_begin(h, PH_GEMM, st);
    e = fault_launch();
    if (e == cudaSuccess) e = launch_gemm_I_tc(p, out_mode, a, st, 1);
    trace_end(h, PH_GEMM, st, 1);
    if (e != cudaSuccess) return cuda_err(e);
    trace_begin(h, PH_OTHER, st);
    e = launch_gemm_I_tc(p, out_mode, a, st, 2);
    trace_end(h, PH_OTHER, st, 1);
    if (e != cudaSuccess) return cuda_err(e);
  }
  return EMU_OK;
}
template emu_status_t run_tri<double>(emu_handle_s*, const View&, int64_t, int, double, double, void*, int64_t, int,
                                      cudaStream_t, uint8_t*, int64_t, int);
template emu_status_t run_tri<float>(emu_handle_s*, const View&, int64_t, int, double, double, void*, int64_t, int,
                                     cudaStream_t, uint8_t*, int64_t, int);

template <typename T>
emu_status_t run_scheme_I(emu_handle_s* h, const View& v, int64_t k, int p, double alpha, double beta,
                          void* C, int64_t ldc, int out_mode, int32_t* partials, cudaStream_t st,
                          uint8_t* ws_override, bool f8, size_t ws_limit) {
  // INT8 slices on the bf16 tensor cores, if the workspace is there: a
  // caller's workspace or fixed scratch of the INT8 kernel's size, a handle
  // that may not grow inside a capture, or memory too full for the planes
  // keeps the INT8 kernel (the same bits).
  const int64_t tri = f8 || out_mode == OUT_PARTIALS ? 0 : tri_rows(v.M, v.N, k, p);
  if (tri > 0) {
    const size_t need = plan_tri(tri, v.N, k, p).bytes;
    uint8_t* tws = ws_override;
    if (tws ? need <= ws_limit : handle_workspace(h, need, st, &tws, true) == EMU_OK)
      return run_tri<T>(h, v, k, p, alpha, beta, C, ldc, out_mode, st, tws, tri, 0);
  }
  Plan pl = plan_I(v.M, v.N, k, p);
  uint8_t* ws = ws_override;
  if (!ws) {
    emu_status_t s = handle_workspace(h, pl.bytes, st, &ws);
    if (s != EMU_OK) return s;
  }
  auto* maxA = reinterpret_cast<unsigned long long*>(ws + pl.off_maxA);
  auto* maxB = reinterpret_cast<unsigned long long*>(ws + pl.off_maxB);
  auto* EA = reinterpret_cast<int32_t*>(ws + pl.off_EA);
  auto* FB = reinterpret_cast<int32_t*>(ws + pl.off_FB);
  auto* hatA = reinterpret_cast<int8_t*>(ws + pl.off_hatA);
  auto* hatB = reinterpret_cast<int8_t*>(ws + pl.off_hatB);
  const T* A = static_cast<const T*>(v.A);
  const T* B = static_cast<const T*>(v.B);
  cudaError_t e = cudaSuccess;
  if (!v.maxA) {
    trace_begin(h, PH_SCAN, st);
    e = launch_zero(ws + pl.off_maxA, pl.off_maxB + sizeof(*maxB) * v.N - pl.off_maxA, st);
    if (e == cudaSuccess)
      e = launch_scan<T>(A, v.ldA, v.a_kcontig, v.M, maxA, B, v.ldB, v.b_kcontig, v.N, maxB, k, 1, true, h->status, st);
    trace_end(h, PH_SCAN, st, 2);
    if (e != cudaSuccess) return cuda_err(e);
  }
  trace_begin(h, PH_SPLIT, st);
  e = launch_split_I<T>(A, v.ldA, v.a_kcontig, v.M, k, p, v.maxA ? v.maxA : maxA, hatA, EA, st, f8);
  if (e == cudaSuccess)
    e = launch_split_I<T>(B, v.ldB, v.b_kcontig, v.N, k, p, v.maxB ? v.maxB : maxB, hatB, FB, st, f8);
  trace_end(h, PH_SPLIT, st, 2);
  if (e != cudaSuccess) return cuda_err(e);
  return scheme_I_gemm(h, hatA, pl.rows_a, hatB, pl.rows_b, pl.cols, v.M, v.N, k, p, EA, FB, alpha, beta, C, ldc,
                       out_mode, partials, st, f8);
}

// The fused Scheme I GEMM on split operands: hatA (rows_a padded rows) and
// hatB (rows_b) in the interleaved slice layout, `cols` bytes per row; C
// (M x N, leading dimension ldc) from the exact slice sums scaled by EA (M)
// and FB (N).
emu_status_t scheme_I_gemm(emu_handle_s* h, const int8_t* hatA, int64_t rows_a, const int8_t* hatB, int64_t rows_b,
                           int64_t cols, int64_t M, int64_t N, int64_t k, int p, const int32_t* EA,
                           const int32_t* FB, double alpha, double beta, void* C, int64_t ldc, int out_mode,
                           int32_t* partials, cudaStream_t st, bool f8) {
  // E4M3 slices run on the tcgen05 kernel (A boxes of 128 B x 128 rows);
  // the INT8 engine uses the mma.sync kernel (32 B x 64 rows).
  const bool tc = f8 && !f8_engine_mma();
  CUtensorMap ta, tb;
  if (!make_tmap_i8(&ta, hatA, static_cast<uint64_t>(cols), static_cast<uint64_t>(rows_a),
                    tc ? 128u : 64u, tc ? 128 : 32) ||
      !make_tmap_i8(&tb, hatB, static_cast<uint64_t>(cols), static_cast<uint64_t>(rows_b), 32))
    return tmap_err();
  GemmIArgs a{};
  a.descA = &ta;
  a.descB = &tb;
  a.M = static_cast<int>(M);
  a.N = static_cast<int>(N);
  a.nk32 = static_cast<int>((k + 31) / 32);
  a.kc32 = static_cast<int>((f8 ? host_chunk_len_F8(p) : host_chunk_len_I(p)) / 32);
  a.EA = EA;
  a.FB = FB;
  a.alpha = alpha;
  a.beta = beta;
  a.C = C;
  a.ldc = ldc;
  a.partials = partials;
  a.status = h->status;
  a.num_sms = h->num_sms;
  trace_begin(h, PH_GEMM, st);
  cudaError_t e = fault_launch();
  if (e == cudaSuccess) e = tc ? launch_gemm_f8tc(p, out_mode, a, st) : launch_gemm_I(p, out_mode, a, st, f8);
  trace_end(h, PH_GEMM, st, 1);
  return cuda_err(e);
}
template emu_status_t run_scheme_I<double>(emu_handle_s*, const View&, int64_t, int, double, double,
                                           void*, int64_t, int, int32_t*, cudaStream_t, uint8_t*, bool, size_t);
template emu_status_t run_scheme_I<float>(emu_handle_s*, const View&, int64_t, int, double, double,
                                          void*, int64_t, int, int32_t*, cudaStream_t, uint8_t*, bool, size_t);

template <typename T>
// Phases (declared in emu_handle.h): B's split once, then A in row chunks
// (per-row scaling makes the chunks independent).
emu_status_t run_scheme_II(emu_handle_s* h, const View& v, int64_t k, int nm, int cw, double ar,
                           double ai, double br, double bi, void* C, int64_t ldc, int out_mode,
                           uint8_t* residues, cudaStream_t st, bool norm, int phase, int64_t plan_rows) {
  const int nsets = cw == 2 ? 3 : 1;
  // the tcgen05 kernel takes bf16 residue planes; the INT8 kernel sums a
  // modulus's products over the whole K in INT32 (|sum| <= k 2^14)
  const bool tc = out_mode != II_RESIDUES && ii_engine_tc();
  if (!tc && k > EMU_K_MAX_II) return EMU_ERR_UNSUPPORTED;
  Plan pl = plan_II(plan_rows > 0 ? plan_rows : v.M, v.N, k, nm, nsets, tc ? 2 : 1);
  pl.rows_a = split_rows(v.M);  // A's planes are laid out for this call's rows
  uint8_t* ws = nullptr;
  emu_status_t s = handle_workspace(h, pl.bytes, st, &ws);
  if (s != EMU_OK) return s;
  auto* maxA = reinterpret_cast<unsigned long long*>(ws + pl.off_maxA);
  auto* maxB = reinterpret_cast<unsigned long long*>(ws + pl.off_maxB);
  auto* EA = reinterpret_cast<int32_t*>(ws + pl.off_EA);
  auto* FB = reinterpret_cast<int32_t*>(ws + pl.off_FB);
  auto* resA = reinterpret_cast<int8_t*>(ws + pl.off_hatA);
  auto* resB = reinterpret_cast<int8_t*>(ws + pl.off_hatB);
  const T* A = static_cast<const T*>(v.A);
  const T* B = static_cast<const T*>(v.B);
  // worst-case scaling (one b for both operands, exponents of the row
  // maxima) or norm-based scaling (hA, hB, exponents of the 2-norms)
  int bA = host_scale_bits_II(nm, k, cw == 2), bB = bA;
  if (norm) host_norm_halves_II(nm, &bA, &bB);
  auto* accA = reinterpret_cast<unsigned long long*>(ws + pl.off_accA);
  auto* accB = reinterpret_cast<unsigned long long*>(ws + pl.off_accB);
  const MethodTables& tabs = method_tables(nm);
  const ModTables& mt = tabs.mod;
  const bool do_a = phase != 1, do_b = phase != 2;
  trace_begin(h, PH_SCAN, st);
  const unsigned long long* mA = v.maxA ? v.maxA : maxA;
  const unsigned long long* mB = v.maxB ? v.maxB : maxB;
  const bool both = do_a && do_b;
  cudaError_t e = cudaSuccess;
  if (!v.maxA) {
    if (both) {  // maxima, and the sums of squares behind them, in one launch
      const size_t end = norm ? pl.off_accB + 2 * sizeof(*accB) * v.N : pl.off_maxB + sizeof(*maxB) * v.N;
      e = launch_zero(ws + pl.off_maxA, end - pl.off_maxA, st);
    }
    if (e == cudaSuccess)
      e = launch_scan<T>(A, v.ldA, v.a_kcontig, v.M, do_a ? maxA : nullptr, B, v.ldB, v.b_kcontig, v.N,
                         do_b ? maxB : nullptr, k, cw, both, h->status, st);
  }
  if (norm) {
    if (v.maxA || !both) {
      if (e == cudaSuccess && do_a) e = launch_zero(accA, 2 * sizeof(*accA) * v.M, st);
      if (e == cudaSuccess && do_b) e = launch_zero(accB, 2 * sizeof(*accB) * v.N, st);
    }
    if (e == cudaSuccess)
      e = launch_norm<T>(A, v.ldA, v.a_kcontig, v.M, mA, do_a ? accA : nullptr, B, v.ldB, v.b_kcontig, v.N, mB,
                         do_b ? accB : nullptr, k, cw, st);
  }
  trace_end(h, PH_SCAN, st, norm ? 3 : do_a + do_b);
  if (e != cudaSuccess) return cuda_err(e);
  trace_begin(h, PH_SPLIT, st);
  if (do_a)
    e = launch_split_II<T>(A, v.ldA, v.a_kcontig, v.M, k, nm, bA, cw, mt, mA, resA, EA, st, norm ? accA : nullptr, tc);
  if (e == cudaSuccess && do_b)
    e = launch_split_II<T>(B, v.ldB, v.b_kcontig, v.N, k, nm, bB, cw, mt, mB, resB, FB, st, norm ? accB : nullptr, tc);
  trace_end(h, PH_SPLIT, st, do_a + do_b);
  if (e != cudaSuccess) return cuda_err(e);
  if (phase == 1) return EMU_OK;
  CUtensorMap ta, tb;
  // tcgen05: the bf16 planes as bytes, 128-byte (64-element) boxes of 128
  // rows (A) and 256 / cluster rows (B: a CTA pair loads half of each
  // 256-column tile per CTA); INT8: 32-byte boxes of 64 / 32 rows
  const uint64_t row_bytes = static_cast<uint64_t>(pl.cols) * (tc ? 2 : 1);
  const int cluster = tc ? gemm_II_tc_cluster(v.M, k) : 1;
  if (!make_tmap_i8(&ta, resA, row_bytes, static_cast<uint64_t>(pl.rows_a) * nm * nsets,
                    tc ? static_cast<uint32_t>(gemm_II_tc_tile_m()) : 64, tc ? 128 : 32) ||
      !make_tmap_i8(&tb, resB, row_bytes, static_cast<uint64_t>(pl.rows_b) * nm * nsets,
                    tc ? static_cast<uint32_t>(gemm_II_tc_tile_n() / cluster) : 32, tc ? 128 : 32))
    return tmap_err();
  GemmIIArgs a{};
  a.descA = &ta;
  a.descB = &tb;
  a.M = static_cast<int>(v.M);
  a.N = static_cast<int>(v.N);
  a.K = static_cast<int>(k);
  a.nk32 = static_cast<int>(pl.cols / 32);
  a.rowsA_pad = static_cast<int>(pl.rows_a);
  a.rowsB_pad = static_cast<int>(pl.rows_b);
  a.nm = nm;
  a.escale = -(bA + bB);
  a.EA = EA;
  a.FB = FB;
  a.alpha_re = ar;
  a.alpha_im = ai;
  a.beta_re = br;
  a.beta_im = bi;
  a.C = C;
  a.ldc = ldc;
  a.residues = residues;
  a.status = h->status;
  a.num_sms = h->num_sms;
  a.cluster = cluster;
  a.scratch = ws + pl.off_scratch;
  if (!tc) {
    trace_begin(h, PH_GEMM, st);
    e = fault_launch();
    if (e == cudaSuccess) e = launch_gemm_II(out_mode, a, mt, tabs.crt, st);
    trace_end(h, PH_GEMM, st, 1);
    return cuda_err(e);
  }
  // the residue GEMM is the traced GEMM phase, the CRT kernel "other"
  trace_begin(h, PH_GEMM, st);
  e = fault_launch();
  if (e == cudaSuccess) e = launch_gemm_II_tc(out_mode, a, mt, tabs.pair, st, 1);
  trace_end(h, PH_GEMM, st, 1);
  if (e != cudaSuccess) return cuda_err(e);
  trace_begin(h, PH_OTHER, st);
  e = launch_gemm_II_tc(out_mode, a, mt, tabs.pair, st, 2);
  trace_end(h, PH_OTHER, st, 1);
  return cuda_err(e);
}

template emu_status_t run_scheme_II<double>(emu_handle_s*, const View&, int64_t, int, int, double, double, double,
                                            double, void*, int64_t, int, uint8_t*, cudaStream_t, bool, int, int64_t);
template emu_status_t run_scheme_II<float>(emu_handle_s*, const View&, int64_t, int, int, double, double, double,
                                           double, void*, int64_t, int, uint8_t*, cudaStream_t, bool, int, int64_t);

template <typename T>
void launch_scale_c(T* C, int64_t ldc, int64_t M, int64_t N, double beta, cudaStream_t st) {
  int64_t tot = M * N;
  if (tot <= 0) return;
  scale_c_kernel<T><<<static_cast<unsigned>((tot + 255) / 256), 256, 0, st>>>(C, ldc, M, N, beta);
}
template void launch_scale_c<double>(double*, int64_t, int64_t, int64_t, double, cudaStream_t);

}  // namespace emu

// ================================================================ entry points
extern "C" {

emu_status_t emu_workspace_size(emu_scheme_t scheme, int64_t m, int64_t n, int64_t k, int p_or_nm,
                                int is_complex, size_t* bytes) {
  if (!bytes || m < 0 || n < 0 || k < 0) return EMU_ERR_INVALID_ARG;
  if (scheme == EMU_SCHEME_I || scheme == EMU_SCHEME_I_F8) {
    if (p_or_nm < EMU_P_MIN || p_or_nm > EMU_P_MAX) return EMU_ERR_UNSUPPORTED;
    *bytes = is_complex ? workspace_complex_I(m, n, k, p_or_nm, scheme == EMU_SCHEME_I_F8)
                        : workspace_I(m, n, k, p_or_nm, scheme == EMU_SCHEME_I_F8);
    return EMU_OK;
  }
  if (scheme == EMU_SCHEME_II || scheme == EMU_SCHEME_II_NORM) {
    if (p_or_nm < EMU_NM_MIN || p_or_nm > EMU_NM_MAX) return EMU_ERR_UNSUPPORTED;
    *bytes = plan_II(m, n, k, p_or_nm, is_complex ? 3 : 1, ii_engine_tc() ? 2 : 1).bytes;
    return EMU_OK;
  }
  return EMU_ERR_INVALID_ARG;
}

}  // extern "C"

emu_status_t emu::gemm_common(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k,
                                const void* A, int64_t lda, const void* B, int64_t ldb, const void* C,
                                int64_t ldc, emu_scheme_t scheme, int p_or_nm) {
  if (!h) return EMU_ERR_INVALID_ARG;
  if (layout != EMU_ROW_MAJOR && layout != EMU_COL_MAJOR) return EMU_ERR_INVALID_ARG;
  if (m < 0 || n < 0 || k < 0) return EMU_ERR_INVALID_ARG;
  if (m > INT32_MAX / 2 || n > INT32_MAX / 2 || k > (int64_t{1} << 30)) return EMU_ERR_UNSUPPORTED;
  if (!check_lds(layout, m, n, k, lda, ldb, ldc)) return EMU_ERR_INVALID_ARG;
  if (m > 0 && n > 0 && !C) return EMU_ERR_INVALID_ARG;
  if (m > 0 && n > 0 && k > 0 && (!A || !B)) return EMU_ERR_INVALID_ARG;
  if (scheme == EMU_SCHEME_I || scheme == EMU_SCHEME_I_F8) {
    if (p_or_nm < EMU_P_MIN || p_or_nm > EMU_P_MAX) return EMU_ERR_UNSUPPORTED;
  } else if (scheme == EMU_SCHEME_II || scheme == EMU_SCHEME_II_NORM) {
    if (p_or_nm < EMU_NM_MIN || p_or_nm > EMU_NM_MAX) return EMU_ERR_UNSUPPORTED;
    if (k > EMU_K_MAX_II && !ii_engine_tc()) return EMU_ERR_UNSUPPORTED;
  } else {
    return EMU_ERR_INVALID_ARG;
  }
  if (cudaSetDevice(h->device) != cudaSuccess) return EMU_ERR_CUDA;
  return EMU_OK;
}

template <typename T>
static emu_status_t real_gemm(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k,
                              double alpha, const T* A, int64_t lda, const T* B, int64_t ldb,
                              double beta, T* C, int64_t ldc, emu_scheme_t scheme, int p_or_nm,
                              emu_stream_t stream, const unsigned long long* maxA = nullptr,
                              const unsigned long long* maxB = nullptr, int32_t* sums = nullptr) {
  emu_status_t s = gemm_common(h, layout, m, n, k, A, lda, B, ldb, C, ldc, scheme, p_or_nm);
  if (s != EMU_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  View v;
  normalize(layout, m, n, A, lda, B, ldb, &v);
  v.maxA = maxA;
  v.maxB = maxB;
  v.sums = sums;
  if (v.M == 0 || v.N == 0) return EMU_OK;
  if (k == 0) {
    launch_scale_c<T>(C, ldc, v.M, v.N, beta, st);
    return cuda_err(cudaGetLastError());
  }
  const int out = sizeof(T) == 8 ? 0 : 1;
  if (scheme == EMU_SCHEME_I || scheme == EMU_SCHEME_I_F8)
    return run_scheme_I<T>(h, v, k, p_or_nm, alpha, beta, C, ldc, out == 0 ? OUT_F64 : OUT_F32, nullptr,
                           st, nullptr, scheme == EMU_SCHEME_I_F8);
  return run_scheme_II<T>(h, v, k, p_or_nm, 1, alpha, 0.0, beta, 0.0, C, ldc, out == 0 ? II_F64 : II_F32,
                          nullptr, st, scheme == EMU_SCHEME_II_NORM);
}

emu_status_t emu::dgemm_scanned(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, double alpha,
                                const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc,
                                emu_scheme_t scheme, int p_or_nm, const unsigned long long* maxA,
                                const unsigned long long* maxB, int32_t* sums, emu_stream_t stream) {
  return real_gemm<double>(h, layout, m, n, k, alpha, A, lda, B, ldb, 0.0, C, ldc, scheme, p_or_nm, stream, maxA,
                           maxB, sums);
}

extern "C" {

emu_status_t emu_dgemm(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, double alpha,
                       const double* A, int64_t lda, const double* B, int64_t ldb, double beta, double* C,
                       int64_t ldc, emu_scheme_t scheme, int p_or_nm, emu_stream_t stream) {
  return real_gemm<double>(h, layout, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, scheme, p_or_nm, stream);
}

emu_status_t emu_sgemm(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k, float alpha,
                       const float* A, int64_t lda, const float* B, int64_t ldb, float beta, float* C,
                       int64_t ldc, emu_scheme_t scheme, int p_or_nm, emu_stream_t stream) {
  return real_gemm<float>(h, layout, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, scheme, p_or_nm, stream);
}

emu_status_t emu_zgemm(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k,
                       const double* alpha, const double* A, int64_t lda, const double* B, int64_t ldb,
                       const double* beta, double* C, int64_t ldc, emu_scheme_t scheme, int nm,
                       emu_stream_t stream) {
  if (!alpha || !beta) return EMU_ERR_INVALID_ARG;
  emu_status_t s = gemm_common(h, layout, m, n, k, A, lda, B, ldb, C, ldc, scheme, nm);
  if (s != EMU_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  View v;
  normalize(layout, m, n, A, lda, B, ldb, &v);
  if (v.M == 0 || v.N == 0) return EMU_OK;
  if (k == 0) {
    int64_t tot = v.M * v.N;
    scale_z_kernel<double>
        <<<static_cast<unsigned>((tot + 255) / 256), 256, 0, st>>>(C, ldc, v.M, v.N, beta[0], beta[1]);
    return cuda_err(cudaGetLastError());
  }
  if (scheme == EMU_SCHEME_I || scheme == EMU_SCHEME_I_F8)
    return run_complex_I<double>(h, layout, m, n, k, A, lda, B, ldb, nm, scheme == EMU_SCHEME_I_F8, alpha, beta,
                                 C, ldc, st);
  return run_scheme_II<double>(h, v, k, nm, 2, alpha[0], alpha[1], beta[0], beta[1], C, ldc, II_Z3M,
                               nullptr, st, scheme == EMU_SCHEME_II_NORM);
}

emu_status_t emu_cgemm(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k,
                       const float* alpha, const float* A, int64_t lda, const float* B, int64_t ldb,
                       const float* beta, float* C, int64_t ldc, emu_scheme_t scheme, int p_or_nm,
                       emu_stream_t stream) {
  if (!alpha || !beta) return EMU_ERR_INVALID_ARG;
  emu_status_t s = gemm_common(h, layout, m, n, k, A, lda, B, ldb, C, ldc, scheme, p_or_nm);
  if (s != EMU_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  View v;
  normalize(layout, m, n, A, lda, B, ldb, &v);
  if (v.M == 0 || v.N == 0) return EMU_OK;
  const double al[2] = {alpha[0], alpha[1]}, be[2] = {beta[0], beta[1]};
  if (k == 0) {
    int64_t tot = v.M * v.N;
    scale_z_kernel<float>
        <<<static_cast<unsigned>((tot + 255) / 256), 256, 0, st>>>(C, ldc, v.M, v.N, be[0], be[1]);
    return cuda_err(cudaGetLastError());
  }
  if (scheme == EMU_SCHEME_II || scheme == EMU_SCHEME_II_NORM)
    return run_scheme_II<float>(h, v, k, p_or_nm, 2, al[0], al[1], be[0], be[1], C, ldc, II_C3M, nullptr, st,
                                scheme == EMU_SCHEME_II_NORM);
  return run_complex_I<float>(h, layout, m, n, k, A, lda, B, ldb, p_or_nm, scheme == EMU_SCHEME_I_F8, al, be, C,
                              ldc, st);
}

// ---------------------------------------------------------------- steps
static emu_status_t split_slices(emu_handle_t h, emu_layout_t layout, int operand, int64_t rows, int64_t k,
                                 const double* X, int64_t ldx, int p, int8_t* hat, int32_t* E, emu_stream_t stream,
                                 bool f8);

emu_status_t emu_split_I(emu_handle_t h, emu_layout_t layout, int operand, int64_t rows, int64_t k,
                         const double* X, int64_t ldx, int p, int8_t* hat, int32_t* E, emu_stream_t stream) {
  return split_slices(h, layout, operand, rows, k, X, ldx, p, hat, E, stream, false);
}

emu_status_t emu_split_F8(emu_handle_t h, emu_layout_t layout, int operand, int64_t rows, int64_t k,
                          const double* X, int64_t ldx, int p, int8_t* hat, int32_t* E, emu_stream_t stream) {
  return split_slices(h, layout, operand, rows, k, X, ldx, p, hat, E, stream, true);
}

}  // extern "C"

static emu_status_t split_slices(emu_handle_t h, emu_layout_t layout, int operand, int64_t rows, int64_t k,
                                 const double* X, int64_t ldx, int p, int8_t* hat, int32_t* E, emu_stream_t stream,
                                 bool f8) {
  if (!h || !hat || !E || rows < 0 || k < 0 || (operand != 0 && operand != 1)) return EMU_ERR_INVALID_ARG;
  if (layout != EMU_ROW_MAJOR && layout != EMU_COL_MAJOR) return EMU_ERR_INVALID_ARG;
  if (p < EMU_P_MIN || p > EMU_P_MAX) return EMU_ERR_UNSUPPORTED;
  if (rows > 0 && k > 0 && !X) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // operand 0: X is rows x k (A); operand 1: X is k x rows (B)
  bool kcontig = (operand == 0) == (layout == EMU_ROW_MAJOR);
  if (ldx < 1) return EMU_ERR_INVALID_ARG;
  uint8_t* ws = nullptr;
  emu_status_t s = handle_workspace(h, 8 * static_cast<size_t>(rows > 0 ? rows : 1), st, &ws);
  if (s != EMU_OK) return s;
  auto* mx = reinterpret_cast<unsigned long long*>(ws);
  cudaError_t e = launch_scan_one<double>(X, ldx, kcontig, rows, k, 1, mx, h->status, st);
  if (e == cudaSuccess) e = launch_split_I<double>(X, ldx, kcontig, rows, k, p, mx, hat, E, st, f8);
  return cuda_err(e);
}

extern "C" {

emu_status_t emu_split_II(emu_handle_t h, emu_layout_t layout, int operand, int64_t rows, int64_t k,
                          int64_t k_total, const double* X, int64_t ldx, int nm, int8_t* res, int32_t* E,
                          emu_stream_t stream) {
  if (!h || !res || !E || rows < 0 || k < 0 || (operand != 0 && operand != 1)) return EMU_ERR_INVALID_ARG;
  if (layout != EMU_ROW_MAJOR && layout != EMU_COL_MAJOR) return EMU_ERR_INVALID_ARG;
  if (nm < EMU_NM_MIN || nm > EMU_NM_MAX) return EMU_ERR_UNSUPPORTED;
  if ((rows > 0 && k > 0 && !X) || ldx < 1) return EMU_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  bool kcontig = (operand == 0) == (layout == EMU_ROW_MAJOR);
  uint8_t* ws = nullptr;
  emu_status_t s = handle_workspace(h, 8 * static_cast<size_t>(rows > 0 ? rows : 1), st, &ws);
  if (s != EMU_OK) return s;
  auto* mx = reinterpret_cast<unsigned long long*>(ws);
  const ModTables& mt = method_tables(nm).mod;
  int b = host_scale_bits_II(nm, k_total, 0);
  cudaError_t e = launch_scan_one<double>(X, ldx, kcontig, rows, k, 1, mx, h->status, st);
  if (e == cudaSuccess) e = launch_split_II<double>(X, ldx, kcontig, rows, k, nm, b, 1, mt, mx, res, E, st);
  return cuda_err(e);
}

emu_status_t emu_partials_I(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k,
                            const double* A, int64_t lda, const double* B, int64_t ldb, int p, int32_t* Cs,
                            emu_stream_t stream) {
  emu_status_t s = gemm_common(h, layout, m, n, k, A, lda, B, ldb, Cs, layout == EMU_ROW_MAJOR ? n : m,
                               EMU_SCHEME_I, p);
  if (s != EMU_OK) return s;
  if (k > host_chunk_len_I(p)) return EMU_ERR_UNSUPPORTED;
  if (layout != EMU_ROW_MAJOR) return EMU_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  View v;
  normalize(layout, m, n, A, lda, B, ldb, &v);
  if (v.M == 0 || v.N == 0) return EMU_OK;
  if (k == 0) return cuda_err(cudaMemsetAsync(Cs, 0, sizeof(int32_t) * p * v.M * v.N, st));
  return run_scheme_I<double>(h, v, k, p, 1.0, 0.0, nullptr, 0, OUT_PARTIALS, Cs, st, nullptr);
}

emu_status_t emu_partials_F8(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k,
                             const double* A, int64_t lda, const double* B, int64_t ldb, int p, int32_t* Cs,
                             emu_stream_t stream) {
  emu_status_t s = gemm_common(h, layout, m, n, k, A, lda, B, ldb, Cs, layout == EMU_ROW_MAJOR ? n : m,
                               EMU_SCHEME_I_F8, p);
  if (s != EMU_OK) return s;
  if (k > host_chunk_len_F8(p)) return EMU_ERR_UNSUPPORTED;
  if (layout != EMU_ROW_MAJOR) return EMU_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  View v;
  normalize(layout, m, n, A, lda, B, ldb, &v);
  if (v.M == 0 || v.N == 0) return EMU_OK;
  if (k == 0) return cuda_err(cudaMemsetAsync(Cs, 0, sizeof(int32_t) * p * v.M * v.N, st));
  return run_scheme_I<double>(h, v, k, p, 1.0, 0.0, nullptr, 0, OUT_PARTIALS, Cs, st, nullptr, true);
}

emu_status_t emu_residues_II(emu_handle_t h, emu_layout_t layout, int64_t m, int64_t n, int64_t k,
                             const double* A, int64_t lda, const double* B, int64_t ldb, int nm, uint8_t* R,
                             emu_stream_t stream) {
  emu_status_t s = gemm_common(h, layout, m, n, k, A, lda, B, ldb, R, layout == EMU_ROW_MAJOR ? n : m,
                               EMU_SCHEME_II, nm);
  if (s != EMU_OK) return s;
  if (layout != EMU_ROW_MAJOR) return EMU_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  View v;
  normalize(layout, m, n, A, lda, B, ldb, &v);
  if (v.M == 0 || v.N == 0) return EMU_OK;
  if (k == 0) return cuda_err(cudaMemsetAsync(R, 0, static_cast<size_t>(nm) * v.M * v.N, st));
  return run_scheme_II<double>(h, v, k, nm, 1, 1.0, 0.0, 0.0, 0.0, nullptr, 0, II_RESIDUES, R, st);
}

}  // extern "C"
