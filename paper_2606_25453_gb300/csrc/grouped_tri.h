// grouped_tri.h -- grouped Scheme I products as bf16 digit triangles
// (grouped_tri.cu), planned and launched by grouped.cu.
#pragma once
#include <vector>

#include "emu_handle.h"
#include "emu_internal.h"

namespace emu {

constexpr int kGroupTriMaxP = 8;

// Last product whose first block is not beyond blk, by the whole warp: 32
// starts per step, so two dependent loads for up to 1024 products.
__device__ __forceinline__ int find_prob(const int* start, int count, int blk) {
  const int lane = threadIdx.x & 31;
  int lo = 0, n = count;
  while (n > 1) {
    const int step = (n + 31) / 32;
    const unsigned in = __ballot_sync(0xFFFFFFFFu, lane * step < n && __ldg(start + lo + min(lane * step, n - 1)) <= blk);
    const int j = max(__popc(in) - 1, 0) * step;
    lo += j;
    n = min(step, n - j);
  }
  return lo;
}

struct GTriProb;  // device table entry of one product

struct GroupTri {
  int p = 0, count = 0, num_sms = 0;
  bool one = false;  // one plane pair per output plane, else one group of them
  void* dev = nullptr;
  GTriProb* d_probs = nullptr;
  CUtensorMap* d_maps = nullptr;
  int4* d_items = nullptr;
  int64_t nitems = 0;
  int *d_startA = nullptr, *d_startB = nullptr, *d_startC = nullptr;  // block prefix arrays
  int split_blocks = 0, comb_blocks = 0;
  uint8_t* zero = nullptr;  // row and column maxima, digit sums: zeroed by every launch
  size_t zero_bytes = 0;
  std::vector<unsigned long long*> maxA, maxB;  // device, per product
};

// Whether a batch takes this path (every product small enough in K, the
// workspace bounded).
bool group_tri_takes(int count, const emu_gemm_desc_t* d, int p);
// Plan and allocate; EMU_ERR_ALLOC if the device memory is not there.
emu_status_t group_tri_build(emu_handle_s* h, int count, const emu_gemm_desc_t* d, int p, GroupTri* g);
void group_tri_free(GroupTri* g);
// Kernel attributes (not stream work; before a capture).
cudaError_t group_tri_prepare();
// Split, GEMM and combine after the grouped scan filled maxA and maxB.
cudaError_t group_tri_launch(const GroupTri& g, int* status, cudaStream_t st);
constexpr int kGroupTriKernels = 3;

}  // namespace emu
