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
// The pair whose rows it reads: lanes past the last pair repeat that one, with w = 0.
__host__ __device__ __forceinline__ size_t gs_read_pair(size_t p, size_t np) { return p < np - 1 ? p : np - 1; }
// How many of its group's rows r0 .. r0 + rb - 1 it reads in a pass that writes row k - 1 of the k (GS_LAG): that row's
// last pair is another thread's, which writes it in the same sweep, so a lane past the end leaves it alone. (Reading
// no row at all there takes a predicate per row and entry pair: Krylov kernels of a 96^3 solve 341 -> 350 ms.)
__host__ __device__ __forceinline__ int gs_read_rows(bool past_end, int k, int r0, int rb) {
    const int n = k - r0 - (past_end ? 1 : 0);
    return n < 0 ? 0 : (n < rb ? n : rb);
}

// The second projection's coefficients c / alpha are of the size of the first one's rounding, about 1e-13. While all
// of them are at most kSmallC, sum_i c_i v_i over the k <= 64 rows is formed in single precision from the rows' high
// words, up to 16 rows a lane and two additions over the lanes (gs_small); above it in double-float. The roundings
// of c and v_i and of the 16 + 2 operations, 2^-24 each, err by at most (2 + 18) 2^-24 64 kSmallC max |v_i| < 2^-53
// max |v_i| of an entry (of those above 2^-91, FP32's subnormals), so with rows of norm 1 by less than 2^-50 of v_j in
// the 2-norm: below the rounding of the double-float pairs that hold it. That takes 11 of the 36 arithmetic instructions per basis entry out.
constexpr double kSmallC = 9.094947017729282379150390625e-13;   // 2^-40
__host__ __device__ __forceinline__ float gs_small(float c, float v_hi, float sum) { return fmaf(c, v_hi, sum); }

}  // namespace stk
