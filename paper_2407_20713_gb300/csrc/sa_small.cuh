// sa_small.cuh -- host side of the few-chain SA kernel (sa_small.cu).
#pragma once
#include "engine_host.h"

namespace sabr {

// Warps per chain and points a warp evaluates at once.
struct SmallShape {
  int nw = 0, kw = 0;
};
// Whether problems of this kind may run in sa_small_kernel, and in what shape.
bool small_supported(int prec, int model);
SmallShape small_shape(int prec, int n_quotes, long long chains);
// More chains than this fill the GPU without speculation.
long long small_most_chains(int prec);
// Blocks of a problem, its dynamic shared memory, and the most blocks of a
// launch that can be resident together (0 if none).
int small_blocks(const SmallShape& s, int n_chains);
size_t small_smem_bytes(int prec, int model, int Q, int M);
int small_capacity(int prec, int model, const SmallShape& s, size_t smem);
// One cooperative launch runs every level of the listed (problem, block)
// items; blocks of a problem meet at its level ends.
cudaError_t launch_small(int prec, int model, const SmallShape& shape, const ProblemDev* probs, const int4* work,
                         int blocks, size_t smem, unsigned long long wait_ns, cudaStream_t s);

}  // namespace sabr
