// block.cu -- the FP32 level operator of the small levels (Section 2.1, definition of A) with its epilogue in
// one launch and without atomic adds: A x, b - A x, or the Jacobi-Chebyshev step of Section 2.2.1.
//
// On levels of a few thousand cells a launch costs more than its arithmetic, so a step is one launch and
// the arithmetic is spread as thin as it goes: a block completes the nodes with local index 0 or 1 in 2 x 2 x 2 cells
// and computes those cells and the ones before them along each axis (3 x 3 x 3, one warp per
// component). A thread transforms its component to the modes of q2_basis.cuh, leaves
// them in shared memory, takes the 24 that it needs of the other two, and leaves its 27 results there;
// then a thread sums the results of up to 8 cells for four nodes and runs the epilogue, whose
// operands it loaded first of all. The first step of a smoothing from zero, x = c0 dinv b, is formed where
// it is gathered. Bound by the instructions of the warps that share a scheduler (some 900 each), so the
// smallest blocks are the fastest although they compute 27 cells for 8: with 4 x 4 x 4 cells and 12 warps the
// FP32 V-cycle at 8^3 took 135 us, now 107; 12^3 100 -> 84, 16^3 181 -> 154 us.
#include "brick.cuh"
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

constexpr int kOwn = 2, kSide = kOwn + 1;              // owned and computed cells per axis
constexpr int kCells = kSide * kSide * kSide;          // 27
constexpr int kLanes = 32;                             // threads per component
constexpr int kBlockThreads = 3 * kLanes;
static_assert(kBlockThreads >= 2 * 3 * kOwn * kOwn * kOwn, "two threads per owned cell and component");

struct BlockArgs {
    int n, M;
    size_t nodes;
    float h;
    const float* mu;
    const float* src;      // operand x; with ZERO not read: x = d = c0 dinv b
    float* dst;            // EPI_PLAIN: A x; EPI_RESID: b - A x; EPI_CHEB: the new x (not src)
    const float* b;
    const float* dinv;
    float* d;              // EPI_CHEB: the direction, in place
    float c0, c1, c2;
};

// Sum of node (I, J, K) (local index 0 or 1 per axis) of component c's cell `at` over the cells that hold it.
template <int I, int J, int K>
__device__ __forceinline__ float node_sum(const float (&W)[3][27][kLanes], int c, int at) {
    float s = 0.0f;
#pragma unroll
    for (int dk = 0; dk <= (K == 0 ? 1 : 0); ++dk)
#pragma unroll
        for (int dj = 0; dj <= (J == 0 ? 1 : 0); ++dj)
#pragma unroll
            for (int di = 0; di <= (I == 0 ? 1 : 0); ++di)
                s += W[c][(I + 2 * di) + 3 * (J + 2 * dj) + 9 * (K + 2 * dk)][at - di - kSide * (dj + kSide * dk)];
    return s;
}

template <int EPI, bool ZERO>
__global__ void __launch_bounds__(kBlockThreads, 5) k_block(BlockArgs a) {
    __shared__ float W[3][27][kLanes];   // the cells' modes, then their results
    const int n = a.n, M = a.M, t = int(threadIdx.x);
    const int x0 = int(blockIdx.x) * kOwn, y0 = int(blockIdx.y) * kOwn, z0 = int(blockIdx.z) * kOwn;
    // ---- the epilogue's operands: nodes (2 oi + i, 2 oj + j, 2 ok + k) of component oc, k this thread's
    const int k = t / (3 * kOwn * kOwn * kOwn), o = t % (3 * kOwn * kOwn * kOwn), oc = o / (kOwn * kOwn * kOwn);
    const int li = o % kOwn, lj = (o / kOwn) % kOwn, lk = (o / (kOwn * kOwn)) % kOwn;
    const int oi = x0 + li, oj = y0 + lj, ok = z0 + lk;
    const bool own = k < 2 && oi < n && oj < n && ok < n && 2 * ok + k > 0;
    const size_t obase = size_t(oc) * a.nodes + size_t(2 * oi) + size_t(M) * (size_t(2 * oj) + size_t(M) * size_t(2 * ok + k));
    bool live[4];
    float eb[4], ei[4], ed[4], ex[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = q & 1, j = q >> 1;
        live[q] = own && 2 * oi + i > 0 && 2 * oj + j > 0;
        const size_t at = obase + size_t(i + M * j);
        eb[q] = ei[q] = ed[q] = ex[q] = 0.0f;
        if (live[q]) {
            if (EPI != EPI_PLAIN) eb[q] = a.b[at];
            if (EPI == EPI_CHEB) {
                ei[q] = a.dinv[at];
                if (!ZERO && a.c1 != 0.0f) ed[q] = a.d[at];
                if (!ZERO) ex[q] = a.src[at];
            }
        }
    }
    // ---- the cell products
    const int c = t / kLanes, lane = t % kLanes;
    const int ci = x0 + lane % kSide - 1, cj = y0 + (lane / kSide) % kSide - 1, ck = z0 + lane / (kSide * kSide) - 1;
    const bool valid = lane < kCells && ci >= 0 && cj >= 0 && ck >= 0 && ci < n && cj < n && ck < n;
    float u[27];
    {
        const size_t base = valid ? size_t(c) * a.nodes + size_t(2 * ci) + size_t(M) * (size_t(2 * cj) + size_t(M) * size_t(2 * ck)) : 0;
        const float* p = (ZERO ? a.b : a.src) + base;
        const float* di = a.dinv + base;
#pragma unroll
        for (int m = 0; m < 27; ++m) {
            const int i = m % 3, j = m / 3 % 3, kk = m / 9;
            const bool bnd = !valid || (i == 0 && ci == 0) || (i == 2 && ci == n - 1) || (j == 0 && cj == 0) ||
                             (j == 2 && cj == n - 1) || (kk == 0 && ck == 0) || (kk == 2 && ck == n - 1);
            const int at = i + M * (j + M * kk);
            u[m] = bnd ? 0.0f : (ZERO ? a.c0 * (di[at] * p[at]) : p[at]);
        }
    }
    const float s = valid ? a.mu[size_t(ci) + size_t(n) * (size_t(cj) + size_t(n) * ck)] * a.h : 0.0f;
    q2::to_modes3(u);
#pragma unroll
    for (int m = 0; m < 27; ++m) W[c][m][lane] = u[m];
    __syncthreads();
    {
        float u1[27], u2[27], w[27];
        const int c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1;
#pragma unroll
        for (int m = 0; m < 27; ++m) {   // those that modes_A does not use are never loaded
            u1[m] = W[c1][m][lane];
            u2[m] = W[c2][m][lane];
        }
        if (c == 0) q2::modes_A<0>(u, u1, u2, w);
        else if (c == 1) q2::modes_A<1>(u, u1, u2, w);
        else q2::modes_A<2>(u, u1, u2, w);
        __syncthreads();
        q2::from_modes3(w);
#pragma unroll
        for (int m = 0; m < 27; ++m) W[c][m][lane] = w[m] * s;
    }
    __syncthreads();
    // ---- the owned nodes
    const int at = (li + 1) + kSide * ((lj + 1) + kSide * (lk + 1));
    float ax[4];
    if (k == 0) {
        ax[0] = node_sum<0, 0, 0>(W, oc, at);
        ax[1] = node_sum<1, 0, 0>(W, oc, at);
        ax[2] = node_sum<0, 1, 0>(W, oc, at);
        ax[3] = node_sum<1, 1, 0>(W, oc, at);
    } else {
        ax[0] = node_sum<0, 0, 1>(W, oc, at);
        ax[1] = node_sum<1, 0, 1>(W, oc, at);
        ax[2] = node_sum<0, 1, 1>(W, oc, at);
        ax[3] = node_sum<1, 1, 1>(W, oc, at);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (!live[q]) continue;
        const size_t i = obase + size_t((q & 1) + M * (q >> 1));
        if (EPI == EPI_PLAIN) {
            a.dst[i] = ax[q];
        } else if (EPI == EPI_RESID) {
            a.dst[i] = eb[q] - ax[q];
        } else {
            if (ZERO) ex[q] = ed[q] = a.c0 * (ei[q] * eb[q]);
            const float dn = (a.c1 != 0.0f ? a.c1 * ed[q] : 0.0f) + a.c2 * (ei[q] * (eb[q] - ax[q]));
            a.d[i] = dn;
            a.dst[i] = ex[q] + dn;
        }
    }
}

}  // namespace

cudaError_t launch_block(int epi, const LevelGeom& g, const float* mu, const float* src, float* dst, const float* b,
                         const float* dinv, float* d, double c0, double c1, double c2, cudaStream_t s) {
    BlockArgs a{};
    a.n = g.n;
    a.M = g.M;
    a.nodes = g.nodes;
    a.h = float(g.h);
    a.mu = mu;
    a.src = src;
    a.dst = dst;
    a.b = b;
    a.dinv = dinv;
    a.d = d;
    a.c0 = float(c0);
    a.c1 = float(c1);
    a.c2 = float(c2);
    const unsigned nb = unsigned((g.n + kOwn - 1) / kOwn);
    const dim3 grid(nb, nb, nb);
    if (epi == EPI_PLAIN) LAUNCH(PROF_VMULT_F32, s, (k_block<EPI_PLAIN, false><<<grid, kBlockThreads, 0, s>>>(a)));
    else if (epi == EPI_RESID) LAUNCH(PROF_VMULT_F32, s, (k_block<EPI_RESID, false><<<grid, kBlockThreads, 0, s>>>(a)));
    else if (src) LAUNCH(PROF_VMULT_F32, s, (k_block<EPI_CHEB, false><<<grid, kBlockThreads, 0, s>>>(a)));
    else LAUNCH(PROF_VMULT_F32, s, (k_block<EPI_CHEB, true><<<grid, kBlockThreads, 0, s>>>(a)));
    return cudaGetLastError();
}

}  // namespace stk
