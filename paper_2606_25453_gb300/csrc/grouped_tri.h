// grouped_tri.h -- grouped Scheme I products as bf16 digit triangles
// (grouped_tri.cu), planned and launched by grouped.cu.
#pragma once
#include <vector>

#include "emu_handle.h"
#include "emu_internal.h"

namespace emu {

constexpr int kGroupTriMaxP = 8;

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
