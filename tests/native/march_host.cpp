// Arguments that the marching level operator (csrc/march.cu) refuses before any device work: its blocks copy
// rows that reach into entries their neighbours write, so a Chebyshev step in place would be a race. Linked
// against the library at load time. Test support only: tests/test_march_host.py.
#include "brick.cuh"

// 1 if a step with these outputs is refused; only in-place ones may be asked (nothing is launched then).
extern "C" int march_refuses(int dst_is_src, int d_new_is_d) {
    using namespace stk;
    if (!dst_is_src && !d_new_is_d) return -1;
    static float v[6][1];   // addresses only
    return launch_march(EPI_CHEB, make_geom(64), v[0], v[1], dst_is_src ? v[1] : v[2], v[3], v[4], v[5],
                        d_new_is_d ? v[5] : v[0], 0.5, 0.5, nullptr) == cudaErrorInvalidValue;
}
