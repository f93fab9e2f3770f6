// sg_batch.h -- the batched-collections kernels (k_batch.cu) and their host
// driver (sg_batch.cpp).  Internal.
#pragma once
#include "sg_internal.h"

namespace sgk {

struct BatchLaunch {
  const float* data;
  const long long* offsets;
  long long nseg;
  long long chunk;          // elements per work item
  long long capacity;       // chunk partials the scratch holds
  int grid;                 // persistent CTAs
  Prog prog;
  int depth;
  void* scratch;
  double* sums;
  long long* first_viol;
  long long* kept;
  unsigned* host_flag;      // pinned: bit 0 violation, bit 1 capacity overflow
  cudaKernel_t jit;         // run-time specialised kernel, or nullptr (interpreter)
};

// with_pre: the precondition is evaluated (contract mode PRE or above)
bool build_chain_prog(const sg_chain& ch, Prog* pr, int* depth, bool with_pre = true);
size_t batch_scratch_bytes(long long nseg, long long capacity);
cudaError_t launch_batch(const BatchLaunch& L, cudaStream_t s, Prof* prof);
int batch_blocks_per_sm(int depth);

// What the schedule chooser needs of the lengths L_i = off[i + 1] - off[i]:
// sums of log2(L_i + 1) and of its square (fixed order), the extremes, the total
// and whether a length is negative.  out and the work space (zeroed once by
// the caller, left zeroed where it must be) on the device.
struct BatchLengths {
  double s, s2;
  long long mn, mx, total;
  int negative, pad;
};
constexpr int kStatCtas = 128;
constexpr size_t kStatWorkBytes = 256 + kStatCtas * sizeof(BatchLengths);
cudaError_t launch_batch_lengths(const long long* off, long long nseg, void* work,
                                 BatchLengths* out, cudaStream_t s);

}  // namespace sgk
