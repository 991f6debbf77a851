// outer.cu -- launcher of the component-split fixed-point outer Stokes blocks (outer.cuh).
#include "internal.cuh"
#include "outer.cuh"
#include "prof.cuh"

#define LAUNCH(cls, s, ...)              \
    do {                                \
        prof_begin((cls), (s));         \
        __VA_ARGS__;                    \
        prof_end((cls), (s));           \
        prof_count(1);                  \
    } while (0)

namespace stk {

namespace {

// Bound by the integer pipes: ~13,400 thread instructions per cell, and the FP64 atomic adds of its 81 + 8
// results. The whole operator (with the clearing of its output) at 64^3: 197 us, at 20^3: 23.6 us; in
// double-float pairs through the Gauss points 854 and 62 us. A alone at 40^3: 44 us; one thread per
// cell with FP64 instructions in the same modes 166 us. 5 CTAs per SM: 128 registers without spills.
template <bool DO_A, bool DO_BT, bool DO_B>
__global__ void __launch_bounds__(kOuterThreads, 5) k_outer_fix(OuterArgs a) {
    __shared__ OuterShared sh;
    const int c = threadIdx.x / kOuterCells, g = threadIdx.x % kOuterCells;
    {
        double T[27];
        outer_phase1<DO_A, DO_B, DO_BT>(a, c, blockIdx.x, g, sh, T, T);
        __syncthreads();
        outer_phase1b<DO_A, DO_B, DO_BT>(a, c, blockIdx.x, g, sh, T);
    }
    __syncthreads();
    double W[27];
    outer_phase2<DO_A, DO_BT, DO_B>(a, c, blockIdx.x, g, sh, W);
}

}  // namespace

cudaError_t launch_outer_fix(const LevelGeom& g, const double* mu, const double* src_u, const double* src_p,
                             double* dst_u, double* dst_p, bool do_a, bool do_bt, bool do_b, cudaStream_t s) {
    OuterArgs a{g.n, g.M, g.nodes, g.h, mu, src_u, src_p, dst_u, dst_p};
    const unsigned nb = unsigned((g.cells + kOuterCells - 1) / kOuterCells);
    if (do_a && do_bt && do_b)
        LAUNCH(PROF_STOKES_F64, s, (k_outer_fix<true, true, true><<<nb, kOuterThreads, 0, s>>>(a)));
    else if (do_a && !do_bt && !do_b)
        LAUNCH(PROF_VMULT_F64, s, (k_outer_fix<true, false, false><<<nb, kOuterThreads, 0, s>>>(a)));
    else if (!do_a && !do_bt && do_b)
        LAUNCH(PROF_STOKES_F64, s, (k_outer_fix<false, false, true><<<nb, kOuterThreads, 0, s>>>(a)));
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

}  // namespace stk
