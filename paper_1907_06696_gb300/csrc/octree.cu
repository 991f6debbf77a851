// octree.cu -- device kernels of the adaptive (octree) path: level operators on the cells of
// one level through an index map (local smoothing, Section 2.2.1 by citation), Q2 transfers
// between levels, copies between the active space and the levels, and the active Stokes
// blocks with hanging-node constraints resolved in the gather and the scatter (Section 2.1,
// with the constrained space of the adaptive meshes).
//
// A thread takes one cell, one node, or (FP64 operators) one component of a cell. Level vectors are component-blocked
// [3][nn]; the active velocity vector is [3][nu] and the active pressure vector [np].
#include "octree.cuh"
#include "outer.cuh"
#include "prof.cuh"
#include "q2_basis.cuh"

#define LAUNCH(cls, s, ...)              \
    do {                                \
        prof_begin((cls), (s));         \
        __VA_ARGS__;                    \
        prof_end((cls), (s));           \
        prof_count(1);                  \
    } while (0)

namespace stk {

namespace {

inline unsigned blocks_for(size_t n, int t) {
    const size_t b = (n + t - 1) / t;
    return unsigned(b == 0 ? 1 : b);
}

// Quadratic Lagrange basis on {0, 1/2, 1} at position p/4 of a parent cell: the three weights of an axis.
// They and their products over the axes are exact in either precision.
template <typename T>
__device__ __forceinline__ void q2_at(int p, T (&w)[3]) {
    w[0] = p == 0 ? T(1) : (p == 1 ? T(0.375) : (p == 3 ? T(-0.125) : T(0)));
    w[1] = p == 1 || p == 3 ? T(0.75) : (p == 2 ? T(1) : T(0));
    w[2] = p == 4 ? T(1) : (p == 1 ? T(-0.125) : (p == 3 ? T(0.375) : T(0)));
}

// Is entry v, read at position `at` of table t, below `bound`? STOKES_DEBUG builds check and record
// the first failure (flag, table + 1, position); release builds return true without a test.
__device__ __forceinline__ bool idx_ok(const OctDebug& d, int t, long long v, long long bound, size_t at) {
#ifdef STOKES_DEBUG
    if (v >= 0 && v < bound - d.cut[t]) return true;
    if (d.status) {
        atomicOr(d.status, kStatusBadIndex);
        if (atomicCAS(d.status + 1, 0u, unsigned(t + 1)) == 0u) {
            d.status[2] = unsigned(uint64_t(at) & 0xffffffffu);
            d.status[3] = unsigned(uint64_t(at) >> 32);
        }
    }
    return false;
#else
    (void)d; (void)t; (void)v; (void)bound; (void)at;
    return true;
#endif
}

// acc += A_l src over the cells of an FP32 level, one thread per cell. Blocks of 64: the gathers and atomic adds of a
// block queue on its SM, and most levels have fewer blocks than the chip has SMs. V-cycle on 3,431 leaves 320 -> 297
// us, 79,080 leaves 671 -> 654 us against blocks of 128; blocks of 32: 302 and 647 us. (Three threads per cell, one
// component each: 328 -> 354 us and 679 -> 776 us with blocks of 128 before.)
constexpr int kCellThreads = 64;
__global__ void __launch_bounds__(kCellThreads) k_oct_cells(OctLevelDev L, const float* __restrict__ mu, const float* __restrict__ src,
                                                   float* __restrict__ acc) {
    const int cell = blockIdx.x * blockDim.x + threadIdx.x;
    if (cell >= L.n_cells) return;
    const int32_t* cn = L.cell_nodes + size_t(cell) * 27;
    float u[3][27], w[3][27];
    unsigned skip = 0;   // bit a: node a is a boundary node (or a bad table entry)
#pragma unroll
    for (int a = 0; a < 27; ++a) {
        const int32_t node = cn[a];
        const bool b = !idx_ok(L.dbg, OCT_CELL_NODES, node, (long long)L.nn, size_t(cell) * 27 + a) ||
                       (L.flags[node] & 1) != 0;
        skip |= unsigned(b) << a;
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c][a] = b ? 0.0f : src[c * L.nn + node];
    }
    q2::cell_A(u, w);
    const float s = mu[cell] * float(L.h);
#pragma unroll
    for (int a = 0; a < 27; ++a) {
        if ((skip >> a) & 1u) continue;
        const int32_t node = cn[a];
#pragma unroll
        for (int c = 0; c < 3; ++c) atomicAdd(acc + c * L.nn + node, w[c][a] * s);
    }
}

// The same on an FP64 level, in the fixed point of the outer operator (outer.cuh): one component per thread,
// 32 cells per block. FP64 instructions run at 1/72 of the integer rate: FP64 V-cycle on 3,431 / 79,000 leaves
// 1,452 / 3,584 -> 530 / 1,644 us.
__global__ void __launch_bounds__(kOuterThreads, 5)
    k_oct_cells_fix(OctLevelDev L, const double* __restrict__ mu, const double* __restrict__ src, double* __restrict__ acc) {
    __shared__ int32_t node[27][kOuterCells + 1];   // the block's piece of the index map; -1: a boundary node
    __shared__ OuterShared sh;
    const int C = int(threadIdx.x) / kOuterCells, g = int(threadIdx.x) % kOuterCells;
    const size_t first = size_t(blockIdx.x) * kOuterCells, map = first * 27, end = size_t(L.n_cells) * 27;
    for (int t = threadIdx.x; t < 27 * kOuterCells; t += kOuterThreads) {
        int32_t v = -1;
        if (map + t < end) {
            v = L.cell_nodes[map + t];
            if (!idx_ok(L.dbg, OCT_CELL_NODES, v, (long long)L.nn, map + t) || (L.flags[v] & 1)) v = -1;
        }
        node[t % 27][t / 27] = v;
    }
    __syncthreads();
    // strides of the own frame's axes C, C + 1, C + 2 in the cell's 27 nodes
    const int q0 = C == 0 ? 1 : (C == 1 ? 3 : 9), q1 = C == 0 ? 3 : (C == 1 ? 9 : 1), q2 = C == 0 ? 9 : (C == 1 ? 1 : 3);
    {
        double u[27];
        int e = 0;
#pragma unroll
        for (int m = 0; m < 27; ++m) {
            const int32_t v = node[(m % 3) * q0 + (m / 3 % 3) * q1 + (m / 9) * q2][g];
            u[m] = v < 0 ? 0.0 : src[C * L.nn + v];
            e = max(e, exp_of(__double_as_longlong(u[m])));
        }
        sh.eu[C][g] = e;
        __syncthreads();
        outer_modes<true, false>(C, g, sh, u);
    }
    __syncthreads();
    if (first + g >= size_t(L.n_cells)) return;
    long long Y[27];
    const FixScale s = outer_velocity<true, false>(C, g, sh, mu[first + g], L.h, Y);
#pragma unroll
    for (int m = 0; m < 27; ++m) {
        const int32_t v = node[(m % 3) * q0 + (m / 3 % 3) * q1 + (m / 9) * q2][g];
        if (v >= 0) atomicAdd(acc + C * L.nn + v, fix_out(Y[m], s));
    }
}

template <typename T>
__global__ void k_oct_copy_boundary(OctLevelDev L, const T* __restrict__ src, T* __restrict__ dst) {
    const size_t n = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (n >= L.nn || !(L.flags[n] & 1)) return;
    for (int c = 0; c < 3; ++c) dst[c * L.nn + n] = src[c * L.nn + n];
}

__global__ void k_oct_diag(OctLevelDev L, const double* __restrict__ mu, const double* __restrict__ ref,
                           double* __restrict__ diag) {
    const int cell = blockIdx.x * blockDim.x + threadIdx.x;
    if (cell >= L.n_cells) return;
    const double s = mu[cell] * L.h;
    for (int a = 0; a < 27; ++a) {
        const int32_t node = L.cell_nodes[size_t(cell) * 27 + a];
        if (!idx_ok(L.dbg, OCT_CELL_NODES, node, (long long)L.nn, size_t(cell) * 27 + a)) continue;
        for (int c = 0; c < 3; ++c) atomicAdd(diag + c * L.nn + node, s * ref[c * 27 + a]);
    }
}

__global__ void k_oct_dinv(OctLevelDev L, const double* __restrict__ diag, double* __restrict__ dinv) {
    const size_t n = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (n >= L.nn) return;
    const bool skip = L.flags[n] != 0;
    for (int c = 0; c < 3; ++c) dinv[c * L.nn + n] = skip ? 0.0 : 1.0 / diag[c * L.nn + n];
}

// The parent's 27 nodes, -1 where the weight is 0 (or the entry is bad). All loads before the first use: a transfer
// that looks at one node after the other waits for up to 27 pairs of dependent loads. FP32 V-cycle on 3,431 leaves
// 339 -> 328 us, 79,080 leaves 681 -> 679 us. FP64 levels look at one node after the other: there the products
// with weights of 0 cost more (1,660 -> 1,684 us on 79,080 leaves).
template <typename T>
__device__ __forceinline__ void parent_nodes(const OctLevelDev& C, uint32_t par, const T (&wx)[3], const T (&wy)[3],
                                             const T (&wz)[3], int32_t (&node)[27]) {
    const int32_t* cn = C.cell_nodes + size_t(par) * 27;
#pragma unroll
    for (int b = 0; b < 27; ++b) {
        const bool on = wx[b % 3] != T(0) && wy[b / 3 % 3] != T(0) && wz[b / 9] != T(0);
        node[b] = on ? cn[b] : -1;
    }
#pragma unroll
    for (int b = 0; b < 27; ++b)
        if (node[b] >= 0 && !idx_ok(C.dbg, OCT_CELL_NODES, node[b], (long long)C.nn, size_t(par) * 27 + b)) node[b] = -1;
}

template <typename T>
__global__ void k_oct_prolongate(OctLevelDev F, OctLevelDev C, const T* __restrict__ coarse, T* __restrict__ fine,
                                 bool add) {
    const size_t n = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (n >= F.nn) return;
    if (F.flags[n] & 1) {
        if (!add)
            for (int c = 0; c < 3; ++c) fine[c * F.nn + n] = T(0);
        return;
    }
    const uint32_t par = F.parent[n];
    const int p = F.pos[n], px = p % 5, py = (p / 5) % 5, pz = p / 25;
    T v[3] = {T(0), T(0), T(0)};
    if (idx_ok(F.dbg, OCT_PARENT, par, C.n_cells, n) && idx_ok(F.dbg, OCT_POS, p, 125, n)) {
        T wx[3], wy[3], wz[3];
        q2_at(px, wx);
        q2_at(py, wy);
        q2_at(pz, wz);
        if constexpr (sizeof(T) == 8) {
            const int32_t* cn = C.cell_nodes + size_t(par) * 27;
#pragma unroll
            for (int b = 0; b < 27; ++b) {
                const T w = wx[b % 3] * wy[b / 3 % 3] * wz[b / 9];
                if (w == T(0)) continue;
                const int32_t node = cn[b];
                if (!idx_ok(C.dbg, OCT_CELL_NODES, node, (long long)C.nn, size_t(par) * 27 + b)) continue;
#pragma unroll
                for (int c = 0; c < 3; ++c) v[c] += w * coarse[c * C.nn + node];
            }
        } else {
            int32_t node[27];
            parent_nodes(C, par, wx, wy, wz, node);
#pragma unroll
            for (int b = 0; b < 27; ++b) {
                const T w = wx[b % 3] * wy[b / 3 % 3] * wz[b / 9];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const T x = node[b] >= 0 ? coarse[c * C.nn + node[b]] : T(0);
                    v[c] += w * x;
                }
            }
        }
    }
    for (int c = 0; c < 3; ++c) fine[c * F.nn + n] = (add ? fine[c * F.nn + n] : T(0)) + v[c];
}

template <typename T>
__global__ void k_oct_restrict_add(OctLevelDev F, OctLevelDev C, const T* __restrict__ fine, T* __restrict__ coarse) {
    const size_t n = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (n >= F.nn || (F.flags[n] & 1)) return;
    const uint32_t par = F.parent[n];
    const int p = F.pos[n], px = p % 5, py = (p / 5) % 5, pz = p / 25;
    if (!idx_ok(F.dbg, OCT_PARENT, par, C.n_cells, n) || !idx_ok(F.dbg, OCT_POS, p, 125, n)) return;
    const T f[3] = {fine[n], fine[F.nn + n], fine[2 * F.nn + n]};
    T wx[3], wy[3], wz[3];
    q2_at(px, wx);
    q2_at(py, wy);
    q2_at(pz, wz);
    if constexpr (sizeof(T) == 8) {
        const int32_t* cn = C.cell_nodes + size_t(par) * 27;
#pragma unroll
        for (int b = 0; b < 27; ++b) {
            const T w = wx[b % 3] * wy[b / 3 % 3] * wz[b / 9];
            if (w == T(0)) continue;
            const int32_t node = cn[b];
            if (!idx_ok(C.dbg, OCT_CELL_NODES, node, (long long)C.nn, size_t(par) * 27 + b)) continue;
            if (C.flags[node] & 1) continue;
#pragma unroll
            for (int c = 0; c < 3; ++c) atomicAdd(coarse + c * C.nn + node, w * f[c]);
        }
    } else {
        int32_t node[27];
        parent_nodes(C, par, wx, wy, wz, node);
        uint32_t skip = 0;
#pragma unroll
        for (int b = 0; b < 27; ++b) {
            const unsigned flag = node[b] >= 0 ? C.flags[node[b]] : 1u;
            skip |= (flag & 1u) << b;
        }
#pragma unroll
        for (int b = 0; b < 27; ++b) {
            if ((skip >> b) & 1u) continue;
            const T w = wx[b % 3] * wy[b / 3 % 3] * wz[b / 9];
#pragma unroll
            for (int c = 0; c < 3; ++c) atomicAdd(coarse + c * C.nn + node[b], w * f[c]);
        }
    }
}

template <typename T>
__global__ void k_oct_copy_to_level(size_t n, const int32_t* __restrict__ ai, const int32_t* __restrict__ li,
                                    size_t nu, size_t nn, const double* __restrict__ active, T* __restrict__ level,
                                    OctDebug dbg) {
    const size_t t = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t >= n) return;
    if (!idx_ok(dbg, OCT_COPY_ACTIVE, ai[t], (long long)nu, t) || !idx_ok(dbg, OCT_COPY_LEVEL, li[t], (long long)nn, t))
        return;
    for (int c = 0; c < 3; ++c) level[c * nn + li[t]] = T(active[c * nu + ai[t]]);
}

template <typename T>
__global__ void k_oct_copy_from_level(size_t n, const int32_t* __restrict__ ai, const int32_t* __restrict__ li,
                                      size_t nu, size_t nn, const T* __restrict__ level, double* __restrict__ active,
                                      OctDebug dbg) {
    const size_t t = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t >= n) return;
    if (!idx_ok(dbg, OCT_COPY_ACTIVE, ai[t], (long long)nu, t) || !idx_ok(dbg, OCT_COPY_LEVEL, li[t], (long long)nn, t))
        return;
    for (int c = 0; c < 3; ++c) active[c * nu + ai[t]] = double(level[c * nn + li[t]]);
}

// ---- active blocks with hanging-node constraints
// A reference r read from leaf_u / leaf_p is a node (r >= 0), constraint -r-1 or (velocity) kOctNoRow. The terms of a
// constraint are loaded together, unused ones (-1: no term, or a Dirichlet row) as zero: their addresses do
// not depend on one another.
__device__ __forceinline__ double con_gather_u(const OctActiveDev& a, const double* src, int c, long long k) {
    const int32_t* nd = a.ucon_node + size_t(k) * kOctUCon;
    const double* wt = a.ucon_w + size_t(k) * kOctUCon;
    double v = 0.0;
#pragma unroll
    for (int t = 0; t < kOctUCon; ++t) {
        const int32_t node = nd[t];
        const bool on = node >= 0 && idx_ok(a.dbg, OCT_UCON_NODE, node, (long long)a.nu_nodes, size_t(k) * kOctUCon + t);
        const double x = src[c * a.nu_nodes + (on ? node : 0)];
        if (on) v += wt[t] * x;
    }
    return v;
}
__device__ __forceinline__ void con_scatter_u(const OctActiveDev& a, double* dst, int c, long long k, double v) {
    const int32_t* nd = a.ucon_node + size_t(k) * kOctUCon;
    const double* wt = a.ucon_w + size_t(k) * kOctUCon;
#pragma unroll
    for (int t = 0; t < kOctUCon; ++t) {
        const int32_t node = nd[t];
        const bool on = node >= 0 && idx_ok(a.dbg, OCT_UCON_NODE, node, (long long)a.nu_nodes, size_t(k) * kOctUCon + t);
        if (on) atomicAdd(dst + c * a.nu_nodes + node, wt[t] * v);
    }
}
__device__ __forceinline__ double gather_p(const OctActiveDev& a, const double* src, int32_t r, size_t at) {
    if (r >= 0) return idx_ok(a.dbg, OCT_LEAF_P, r, (long long)a.np, at) ? src[r] : 0.0;
    const long long k = -(long long)r - 1;
    if (!idx_ok(a.dbg, OCT_LEAF_P, k, (long long)a.n_pcon, at)) return 0.0;
    const int32_t* nd = a.pcon_node + size_t(k) * kOctPCon;
    const double* wt = a.pcon_w + size_t(k) * kOctPCon;
    double v = 0.0;
#pragma unroll
    for (int t = 0; t < kOctPCon; ++t) {
        const int32_t node = nd[t];
        const bool on = node >= 0 && idx_ok(a.dbg, OCT_PCON_NODE, node, (long long)a.np, size_t(k) * kOctPCon + t);
        const double x = src[on ? node : 0];
        if (on) v += wt[t] * x;
    }
    return v;
}
__device__ __forceinline__ void scatter_p(const OctActiveDev& a, double* dst, int32_t r, double v, size_t at) {
    if (r >= 0) {
        if (idx_ok(a.dbg, OCT_LEAF_P, r, (long long)a.np, at)) atomicAdd(dst + r, v);
        return;
    }
    const long long k = -(long long)r - 1;
    if (!idx_ok(a.dbg, OCT_LEAF_P, k, (long long)a.n_pcon, at)) return;
    const int32_t* nd = a.pcon_node + size_t(k) * kOctPCon;
    const double* wt = a.pcon_w + size_t(k) * kOctPCon;
#pragma unroll
    for (int t = 0; t < kOctPCon; ++t) {
        const int32_t node = nd[t];
        if (node >= 0 && idx_ok(a.dbg, OCT_PCON_NODE, node, (long long)a.np, size_t(k) * kOctPCon + t))
            atomicAdd(dst + node, wt[t] * v);
    }
}

// The block's references to velocity nodes, and the places of the constrained ones, at * kOuterCells + leaf.
struct OctRefs {
    int32_t u[27][kOuterCells + 1];
    uint16_t hang[27 * kOuterCells];
    int n_hang;
};

// One velocity component per thread, 32 leaves per CTA, in the fixed-point arithmetic of the uniform
// outer operator (outer.cuh): warp c gathers component c through the leaf's references and scatters it the same
// way. A hanging node's value is a chain of dependent loads (constraint, nodes, values). Taken
// where the leaf comes to it, the whole warp waits for the chain at each of the 27 nodes, so the block first
// lists its hanging nodes, one lane takes one of them, and the values go through the (then unused) space of
// the modes in shared memory. 79,080 leaves (with the clearing of the output): 406 -> 170 us, of which the uniform
// operator on as many cells takes some 60.
// On meshes of at most one block per SM the time is that of the block with the most hanging nodes (up to 600,
// 20 rounds of 32 lanes): there GROUPS - 1 more warps per component take part in those rounds alone. Stokes operator on 3,431
// leaves 49.2 -> 32.8 us, with the Dirichlet flags folded into the tables; that alone took this kernel (without the
// clearing and the boundary rows) on 79,080 leaves from 149 to 132 us, the operator to 146 us.
template <bool DO_A, bool DO_BT, bool DO_B, int GROUPS>
__global__ void __launch_bounds__(kOuterThreads * GROUPS, GROUPS == 1 ? 5 : 1)
    k_oct_active(OctActiveDev a, const double* __restrict__ src_u, const double* __restrict__ src_p, double* __restrict__ dst_u,
                 double* __restrict__ dst_p) {
    __shared__ OuterShared sh;
    __shared__ OctRefs ref;
    const int C = int(threadIdx.x) / kOuterCells % 3, g = int(threadIdx.x) % kOuterCells;
    const int group = int(threadIdx.x) / kOuterThreads;
    const int leaf = int(blockIdx.x) * kOuterCells + g;
    const bool main = GROUPS == 1 || group == 0, valid = main && leaf < a.n_leaves;
    const int32_t* rp = a.leaf_p + size_t(valid ? leaf : 0) * 8;
    // strides of the own frame's axes in the leaf's 27 nodes
    const int q0 = C == 0 ? 1 : (C == 1 ? 3 : 9), q1 = C == 0 ? 3 : (C == 1 ? 9 : 1), q2 = C == 0 ? 9 : (C == 1 ? 1 : 3);
    if (threadIdx.x == 0) ref.n_hang = 0;
    __syncthreads();
    const size_t map = size_t(blockIdx.x) * kOuterCells * 27, end = size_t(a.n_leaves) * 27;
#pragma unroll
    for (int t = threadIdx.x; t < 27 * kOuterCells; t += kOuterThreads * GROUPS) {
        int32_t r = kOctNoRow;
        if (map + t < end) {
            r = a.leaf_u[map + t];
            if (r != kOctNoRow && !(r >= 0 ? idx_ok(a.dbg, OCT_LEAF_U, r, (long long)a.nu_nodes, map + t)
                                           : idx_ok(a.dbg, OCT_LEAF_U, -(long long)r - 1, (long long)a.n_ucon, map + t)))
                r = kOctNoRow;
        }
        ref.u[t % 27][t / 27] = r;
        if (r < 0 && r != kOctNoRow) ref.hang[atomicAdd(&ref.n_hang, 1)] = uint16_t(t % 27 * kOuterCells + t / 27);
    }
    __syncthreads();
    const int n_hang = ref.n_hang;
    {
        double T[27];
        if (DO_A || DO_B) {
            for (int i = g + kOuterCells * group; i < n_hang; i += kOuterCells * GROUPS) {
                const int at = ref.hang[i] / kOuterCells, l = ref.hang[i] % kOuterCells;
                sh.U[C][at][l] = __double_as_longlong(con_gather_u(a, src_u, C, -(long long)ref.u[at][l] - 1));
            }
            if (GROUPS == 1) __syncwarp();
            else __syncthreads();
            if (main) {
                int e = 0;
#pragma unroll
                for (int m = 0; m < 27; ++m) {
                    const int at = (m % 3) * q0 + (m / 3 % 3) * q1 + (m / 9) * q2;
                    const int32_t r = ref.u[at][g];
                    T[m] = r >= 0 ? src_u[C * a.nu_nodes + r] : (r == kOctNoRow ? 0.0 : __longlong_as_double(sh.U[C][at][g]));
                    e = max(e, exp_of(__double_as_longlong(T[m])));
                }
                sh.eu[C][g] = e;
            }
        }
        if (DO_BT && main) {
            int e = 0;
            for (int v = C; v < 8; v += 3) {
                const long long b = __double_as_longlong(valid ? gather_p(a, src_p, rp[v], size_t(leaf) * 8 + v) : 0.0);
                e = max(e, exp_of(b));
                sh.P[v][g] = b;
            }
            sh.ep[C][g] = e;
        }
        __syncthreads();
        if (main) outer_modes<DO_A || DO_B, DO_BT>(C, g, sh, T);
    }
    __syncthreads();
    const double h = valid ? ldexp(1.0, -int(a.level[leaf])) : 1.0;
    if (DO_B && valid) {
        long long b[8];
        const FixScale s = outer_pressure(C, g, sh, h, b);
        const int v1 = 1 << C, v6 = 7 - v1;   // as in outer_phase2: each vertex by one warp
        scatter_p(a, dst_p, rp[v1], fix_out(b[1], s), size_t(leaf) * 8 + v1);
        scatter_p(a, dst_p, rp[v6], fix_out(b[6], s), size_t(leaf) * 8 + v6);
        if (C < 2) {
            const int v = C == 0 ? 0 : 7;
            scatter_p(a, dst_p, rp[v], fix_out(C == 0 ? b[0] : b[7], s), size_t(leaf) * 8 + v);
        }
    }
    if (DO_A || DO_BT) {
        long long Y[27];
        FixScale s;
        if (main) s = outer_velocity<DO_A, DO_BT>(C, g, sh, valid ? a.mu[leaf] : 1.0, h, Y);
        __syncthreads();   // every warp has read the modes
        if (main) {
#pragma unroll
            for (int m = 0; m < 27; ++m) {
                const int at = (m % 3) * q0 + (m / 3 % 3) * q1 + (m / 9) * q2;
                const int32_t r = ref.u[at][g];
                const double y = fix_out(Y[m], s);
                if (r >= 0) atomicAdd(dst_u + C * a.nu_nodes + r, y);
                else if (r != kOctNoRow) sh.U[C][at][g] = __double_as_longlong(y);
            }
        }
        if (GROUPS == 1) __syncwarp();
        else __syncthreads();
        for (int i = g + kOuterCells * group; i < n_hang; i += kOuterCells * GROUPS) {
            const int at = ref.hang[i] / kOuterCells, l = ref.hang[i] % kOuterCells;
            con_scatter_u(a, dst_u, C, -(long long)ref.u[at][l] - 1, __longlong_as_double(sh.U[C][at][l]));
        }
    }
}

__global__ void k_oct_active_boundary(OctActiveDev a, const double* __restrict__ src_u, double* __restrict__ dst_u) {
    const size_t n = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (n >= a.nu_nodes || !a.ubnd[n]) return;
    for (int c = 0; c < 3; ++c) dst_u[c * a.nu_nodes + n] = src_u[c * a.nu_nodes + n];
}

// M_p: one thread per vertex of a leaf, the element matrix (2, 1; 1, 2)/6 per axis by exchanges within the leaf's
// 8 lanes. With it and k_oct_active a solve on 3,431 leaves took 97
// instead of 128 ms (one thread per leaf, the 64 products of the matrix).
__global__ void __launch_bounds__(256) k_oct_mass_p(OctActiveDev a, const double* __restrict__ src, double* __restrict__ dst) {
    const size_t t = size_t(blockIdx.x) * blockDim.x + threadIdx.x, end = size_t(a.n_leaves) * 8;
    const int32_t r = t < end ? a.leaf_p[t] : 0;
    double p = t < end ? gather_p(a, src, r, t) * (1.0 / 216.0) : 0.0;
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) p = 2.0 * p + __shfl_xor_sync(0xffffffffu, p, d);
    if (t >= end) return;
    const size_t leaf = t / 8;
    const double h = ldexp(1.0, -int(a.level[leaf]));
    scatter_p(a, dst, r, h * h * h / a.mu[leaf] * p, t);
}

}  // namespace

const char* oct_table_name(int table) {
    static const char* names[OCT_NTABLES] = {"cell_nodes", "parent", "pos", "leaf_u", "ucon_node",
                                             "leaf_p", "pcon_node", "copy_active", "copy_level"};
    return table >= 0 && table < OCT_NTABLES ? names[table] : "?";
}

template <typename T>
cudaError_t launch_oct_level_cells(const OctLevelDev& L, const T* mu, const T* src, T* acc, cudaStream_t s) {
    if (L.n_cells == 0) return cudaSuccess;
    if constexpr (sizeof(T) == 4)
        LAUNCH(PROF_VMULT_F32, s, (k_oct_cells<<<blocks_for(L.n_cells, kCellThreads), kCellThreads, 0, s>>>(L, mu, src, acc)));
    else
        LAUNCH(PROF_VMULT_F64, s, (k_oct_cells_fix<<<blocks_for(L.n_cells, kOuterCells), kOuterThreads, 0, s>>>(L, mu, src, acc)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_oct_copy_boundary(const OctLevelDev& L, const T* src, T* dst, cudaStream_t s) {
    LAUNCH(PROF_SMOOTH_VEC, s, (k_oct_copy_boundary<T><<<blocks_for(L.nn, 256), 256, 0, s>>>(L, src, dst)));
    return cudaGetLastError();
}

cudaError_t launch_oct_inv_diag(const OctLevelDev& L, const double* mu, const double* ref_diag81, double* tmp,
                                double* dinv, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(tmp, 0, 3 * L.nn * sizeof(double), s);
    if (e != cudaSuccess) return e;
    if (L.n_cells) LAUNCH(PROF_SMOOTH_VEC, s, (k_oct_diag<<<blocks_for(L.n_cells, 128), 128, 0, s>>>(L, mu, ref_diag81, tmp)));
    LAUNCH(PROF_SMOOTH_VEC, s, (k_oct_dinv<<<blocks_for(L.nn, 256), 256, 0, s>>>(L, tmp, dinv)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_oct_prolongate(const OctLevelDev& F, const OctLevelDev& C, const T* coarse, T* fine, bool add,
                                  cudaStream_t s) {
    LAUNCH(PROF_TRANSFER, s, (k_oct_prolongate<T><<<blocks_for(F.nn, 128), 128, 0, s>>>(F, C, coarse, fine, add)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_oct_restrict_add(const OctLevelDev& F, const OctLevelDev& C, const T* fine, T* coarse,
                                    cudaStream_t s) {
    LAUNCH(PROF_TRANSFER, s, (k_oct_restrict_add<T><<<blocks_for(F.nn, 128), 128, 0, s>>>(F, C, fine, coarse)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_oct_copy_to_level(size_t n_copy, const int32_t* active_idx, const int32_t* level_idx,
                                     size_t nu_nodes, size_t level_nn, const double* active, T* level,
                                     const OctDebug& dbg, cudaStream_t s) {
    if (n_copy == 0) return cudaSuccess;
    LAUNCH(PROF_CAST, s, (k_oct_copy_to_level<T><<<blocks_for(n_copy, 256), 256, 0, s>>>(
                             n_copy, active_idx, level_idx, nu_nodes, level_nn, active, level, dbg)));
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_oct_copy_from_level(size_t n_copy, const int32_t* active_idx, const int32_t* level_idx,
                                       size_t nu_nodes, size_t level_nn, const T* level, double* active,
                                       const OctDebug& dbg, cudaStream_t s) {
    if (n_copy == 0) return cudaSuccess;
    LAUNCH(PROF_CAST, s, (k_oct_copy_from_level<T><<<blocks_for(n_copy, 256), 256, 0, s>>>(
                             n_copy, active_idx, level_idx, nu_nodes, level_nn, level, active, dbg)));
    return cudaGetLastError();
}

namespace {

template <bool DO_A, bool DO_BT, bool DO_B>
void launch_active(int cls, const OctActiveDev& a, const double* src_u, const double* src_p, double* dst_u, double* dst_p,
                   cudaStream_t s) {
    constexpr int kWide = 4, kSms = 152;
    const unsigned n = blocks_for(a.n_leaves, kOuterCells);
    if (n <= kSms)
        LAUNCH(cls, s, (k_oct_active<DO_A, DO_BT, DO_B, kWide><<<n, kWide * kOuterThreads, 0, s>>>(a, src_u, src_p, dst_u, dst_p)));
    else
        LAUNCH(cls, s, (k_oct_active<DO_A, DO_BT, DO_B, 1><<<n, kOuterThreads, 0, s>>>(a, src_u, src_p, dst_u, dst_p)));
}

}  // namespace

cudaError_t launch_oct_active(const OctActiveDev& a, const double* src_u, const double* src_p, double* dst_u,
                              double* dst_p, bool do_a, bool do_bt, bool do_b, cudaStream_t s) {
    cudaError_t e;
    if ((do_a || do_bt) && (e = cudaMemsetAsync(dst_u, 0, 3 * a.nu_nodes * sizeof(double), s)) != cudaSuccess) return e;
    if (do_b && (e = cudaMemsetAsync(dst_p, 0, a.np * sizeof(double), s)) != cudaSuccess) return e;
    const int cls = do_a ? PROF_STOKES_F64 : (do_bt ? PROF_BT_F64 : PROF_STOKES_F64);
    if (do_a && do_bt && do_b) launch_active<true, true, true>(cls, a, src_u, src_p, dst_u, dst_p, s);
    else if (do_a && !do_bt && !do_b) launch_active<true, false, false>(cls, a, src_u, src_p, dst_u, dst_p, s);
    else if (!do_a && do_bt && !do_b) launch_active<false, true, false>(cls, a, src_u, src_p, dst_u, dst_p, s);
    else if (!do_a && !do_bt && do_b) launch_active<false, false, true>(cls, a, src_u, src_p, dst_u, dst_p, s);
    else return cudaErrorInvalidValue;
    if (do_a) LAUNCH(cls, s, (k_oct_active_boundary<<<blocks_for(a.nu_nodes, 256), 256, 0, s>>>(a, src_u, dst_u)));
    return cudaGetLastError();
}

cudaError_t launch_oct_identity_rows(const OctActiveDev& a, const double* src_u, double* dst_u, cudaStream_t s) {
    LAUNCH(PROF_SMOOTH_VEC, s, (k_oct_active_boundary<<<blocks_for(a.nu_nodes, 256), 256, 0, s>>>(a, src_u, dst_u)));
    return cudaGetLastError();
}

cudaError_t launch_oct_mass_p(const OctActiveDev& a, const double* src, double* dst, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(dst, 0, a.np * sizeof(double), s);
    if (e != cudaSuccess) return e;
    LAUNCH(PROF_MASS_P, s, (k_oct_mass_p<<<blocks_for(size_t(a.n_leaves) * 8, 256), 256, 0, s>>>(a, src, dst)));
    return cudaGetLastError();
}

#define INST(T)                                                                                                     \
    template cudaError_t launch_oct_level_cells<T>(const OctLevelDev&, const T*, const T*, T*, cudaStream_t);      \
    template cudaError_t launch_oct_copy_boundary<T>(const OctLevelDev&, const T*, T*, cudaStream_t);              \
    template cudaError_t launch_oct_prolongate<T>(const OctLevelDev&, const OctLevelDev&, const T*, T*, bool,      \
                                                  cudaStream_t);                                                  \
    template cudaError_t launch_oct_restrict_add<T>(const OctLevelDev&, const OctLevelDev&, const T*, T*,          \
                                                    cudaStream_t);                                                \
    template cudaError_t launch_oct_copy_to_level<T>(size_t, const int32_t*, const int32_t*, size_t, size_t,       \
                                                     const double*, T*, const OctDebug&, cudaStream_t);           \
    template cudaError_t launch_oct_copy_from_level<T>(size_t, const int32_t*, const int32_t*, size_t, size_t,     \
                                                       const T*, double*, const OctDebug&, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace stk
