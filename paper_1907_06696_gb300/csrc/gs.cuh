// gs.cuh -- rules of the double-float Gram-Schmidt passes (krylov.cu) as plain functions, so that a host
// program can walk through them.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace stk {

constexpr int kGsThreads = 128;

// Entry pair of a thread in the sweep that starts at `base`, tpe adjacent threads to a pair.
__host__ __device__ __forceinline__ size_t gs_pair(size_t base, unsigned block, int thread, int tpe) {
    return base + size_t(block) * unsigned(kGsThreads / tpe) + unsigned(thread / tpe);
}
// Whether the thread reads the basis rows at its pair p of np where the pass writes one of them (GS_LAG, row j): past
// the end there is nothing to read, the last pair is another thread's, which writes it in the same sweep.
__host__ __device__ __forceinline__ bool gs_reads(size_t p, size_t np) { return p < np; }

}  // namespace stk
