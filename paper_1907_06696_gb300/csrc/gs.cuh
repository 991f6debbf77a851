// gs.cuh -- rules of the double-float Gram-Schmidt passes (krylov.cu) as plain functions, so that a host
// program can walk through them.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
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

// The second projection's coefficients c / alpha are of the size of the first one's rounding, about 1e-13. While all
// of them are at most kSmallC, sum_i c_i v_i over the k <= 64 rows is formed in single precision from the rows' high
// words, up to 16 rows a lane and two additions over the lanes (gs_small); above it in double-float. The roundings
// of c and v_i and of the 16 + 2 operations, 2^-24 each, err by at most (2 + 18) 2^-24 64 kSmallC max |v_i| < 2^-53
// max |v_i| of an entry (of those above 2^-91, FP32's subnormals), so with rows of norm 1 by less than 2^-50 of v_j in
// the 2-norm: below the rounding of the double-float pairs that hold it. That takes 11 of the 36 arithmetic instructions per basis entry out.
constexpr double kSmallC = 9.094947017729282379150390625e-13;   // 2^-40
__host__ __device__ __forceinline__ float gs_small(float c, float v_hi, float sum) { return fmaf(c, v_hi, sum); }

}  // namespace stk
