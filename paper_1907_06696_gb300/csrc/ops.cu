// ops.cu -- matrix-free Q2-Q1 operators and the set-up kernels.
//
// The FP64 outer operator [A, B^T; B, 0] (Section 2.1): the fixed-point kernel of outer.cuh adds the
//   cells' contributions into the zeroed outputs; constrained (boundary-node) rows then get src.
// M_p (Section 2.2.2): Q1 mass matrix weighted by 1/mu per cell.
// Set-up: viscosity at the Gauss points and its harmonic cell average
//   (Section 2.3), Q0 restriction (parent = mean of children, Section 2.3),
//   the sinker right-hand side (Section 3.2), diagonals.
#include "internal.cuh"
#include "q2_basis.cuh"
#include "df64.cuh"
#include "prof.cuh"
#include "pressure.cuh"

#define LAUNCH(cls, s, ...)              \
    do {                                \
        prof_begin((cls), (s));         \
        __VA_ARGS__;                    \
        prof_end((cls), (s));           \
        prof_count(1);                  \
    } while (0)

namespace stk {

namespace {

__device__ __forceinline__ bool on_bnd(int gi, int M) { return gi == 0 || gi == M - 1; }

// Boundary nodes of an M^3 lattice: 6 faces of M*M nodes (edges repeated; writes are identical).
template <typename T>
__global__ void k_copy_boundary(int M, const T* __restrict__ in, T* __restrict__ out) {
    const size_t t = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const size_t face = size_t(M) * M;
    if (t >= 6 * face) return;
    const int f = int(t / face);
    const int a = int((t % face) % M), b = int((t % face) / M);
    const int fixed = (f & 1) ? M - 1 : 0;
    int i, j, k;
    if (f < 2) { i = fixed; j = a; k = b; } else if (f < 4) { i = a; j = fixed; k = b; } else { i = a; j = b; k = fixed; }
    const size_t nodes = size_t(M) * M * M;
    const size_t node = size_t(i) + size_t(M) * (j + size_t(M) * k);
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c * nodes + node] = in ? in[c * nodes + node] : T(0);
}

// z = x on the free nodes, r on the domain boundary; z may be r.
template <typename T>
__global__ void __launch_bounds__(256) k_free_rows(int M, const T* __restrict__ x, const double* r, double* z) {
    const size_t nodes = size_t(M) * M * M, node = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (node >= nodes) return;
    const bool b = on_bnd(int(node % M), M) || on_bnd(int(node / M % M), M) || on_bnd(int(node / (size_t(M) * M)), M);
#pragma unroll
    for (int c = 0; c < 3; ++c) z[c * nodes + node] = b ? r[c * nodes + node] : double(x[c * nodes + node]);
}

// ---------------------------------------------------------------- pressure mass
__global__ void k_mass_p(int n, double h, const double* __restrict__ mu, const double* __restrict__ src,
                         double* __restrict__ dst) {
    const size_t cell = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const size_t cells = size_t(n) * n * n;
    if (cell >= cells) return;
    const int ci = int(cell % n), cj = int((cell / n) % n), ck = int(cell / (size_t(n) * n));
    const int P = n + 1;
    size_t vert[8];
    double p[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        vert[v] = size_t(ci + (v & 1)) + size_t(P) * (cj + ((v >> 1) & 1) + size_t(P) * (ck + (v >> 2)));
        p[v] = src[vert[v]];
    }
    const double s = h * h * h / mu[cell];
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        double acc = 0.0;
#pragma unroll
        for (int b = 0; b < 8; ++b)
            acc += q2::M1(a & 1, b & 1) * q2::M1((a >> 1) & 1, (b >> 1) & 1) * q2::M1(a >> 2, b >> 2) * p[b];
        atomicAdd(dst + vert[a], s * acc);
    }
}

// ---- B^T on the uniform mesh as a gather, one thread per cell (e, f, g) and its 8 nodes of lower or odd
// index (pressure.cuh bt_nodes); nodes on the domain boundary are left as they are.
// BT_PLAIN: out = B^T p;  BT_RESID: out = r - B^T p (the V-cycle's right-hand side), TO = double in FP64,
// TO = float (the right-hand side of an FP32 V-cycle) in double-float without an FP64 instruction, or in FP64 where
// the caller asked for that arithmetic (outer_arith = 0), rounded once at the end.
// Bound by memory (r read, out written) and, in FP64, by its ~3 FP64 instructions per node. At 64^3 the
// fused FP32 right-hand side takes 38 us; one thread per vertex of a line and component, with the moments
// as double-float weights, took 101 us for B^T p alone, 49 us for the FP64 block now.
enum BtMode { BT_PLAIN = 0, BT_RESID = 1 };

template <typename TO, bool DF>
struct BtArith {
    using type = double;
    static __device__ __forceinline__ double in(double v) { return v; }
    static __device__ __forceinline__ TO out(double v) { return TO(v); }
};
template <> struct BtArith<float, true> {
    using type = q2::df64;
    static __device__ __forceinline__ q2::df64 in(double v) { return q2::split_double(v); }
    static __device__ __forceinline__ float out(const q2::df64& v) { return v.hi; }
};

template <int C, int MODE, typename TO, bool DF>
__device__ __forceinline__ void bt_store(const typename BtArith<TO, DF>::type (&v)[3][3][3], double h, int e, int f, int g, int M,
                                         const double* __restrict__ r, TO* __restrict__ out) {
    using A = BtArith<TO, DF>;
    using T = typename A::type;
    T b[8];
    bt_nodes<C>(v, b);
    const size_t base = size_t(C) * M * M * M + size_t(2 * e) + size_t(M) * (size_t(2 * f) + size_t(M) * size_t(2 * g));
    const T even = A::in(-h * h * bt_factor<0>(0, 0, 0)), odd = A::in(-h * h * bt_factor<0>(1, 0, 0));
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                if ((i == 0 && e == 0) || (j == 0 && f == 0) || (k == 0 && g == 0)) continue;
                const size_t at = base + size_t(i + M * (j + M * k));
                const T y = b[i + 2 * j + 4 * k] * ((C == 0 ? i : (C == 1 ? j : k)) != 0 ? odd : even);
                out[at] = A::out(MODE == BT_RESID ? A::in(r[at]) - y : y);
            }
}

template <int MODE, typename TO, bool DF>
__global__ void __launch_bounds__(128) k_bt(int n, double h, const double* __restrict__ p, const double* __restrict__ r,
                                            TO* __restrict__ out) {
    using A = BtArith<TO, DF>;
    const size_t cell = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= size_t(n) * n * n) return;
    const int e = int(cell % n), f = int((cell / n) % n), g = int(cell / (size_t(n) * n));
    const int P = n + 1, M = 2 * n + 1;
    typename A::type v[3][3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                if ((i == 0) + (j == 0) + (k == 0) > 1) continue;   // not used by any component
                const int a = max(e - 1 + i, 0), b = max(f - 1 + j, 0), c = max(g - 1 + k, 0);
                v[k][j][i] = A::in(p[size_t(a) + size_t(P) * (b + size_t(P) * c)]);
            }
    bt_store<0, MODE, TO, DF>(v, h, e, f, g, M, r, out);
    bt_store<1, MODE, TO, DF>(v, h, e, f, g, M, r, out);
    bt_store<2, MODE, TO, DF>(v, h, e, f, g, M, r, out);
}

// s_K = h^3 / mu_K per cell: the factor of the cell's pressure mass matrix (Section 2.2.2, the
// 1/mu-weighted mass matrix), as k_mass_p forms it.
__global__ void k_mass_scale(size_t cells, double h, const double* __restrict__ mu, double* __restrict__ scale) {
    const size_t cell = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell < cells) scale[cell] = h * h * h / mu[cell];
}

// One Jacobi-Chebyshev step of S_hat^-1 with the M_p product gathered per pressure vertex
// (pressure.cuh schur_sum): no atomics. A block takes 8 x 8 x 4 vertices; their neighbours and the cells
// around them are split to double-float once, into shared memory (a thread on its own splits 27 + 8).
// 64^3: 18.8 us; one thread per vertex with 64 products 33.4 us.
constexpr int kSchurX = 8, kSchurY = 8, kSchurZ = 4;
__global__ void __launch_bounds__(kSchurX* kSchurY* kSchurZ)
    k_schur_cheb(int n, const double* __restrict__ scale, const double* __restrict__ r, const double* __restrict__ dinv,
                 const double* __restrict__ z, const double* __restrict__ d, double* __restrict__ z_new,
                 double* __restrict__ d_new, double c1, double c2) {
    __shared__ q2::df64 zt[kSchurZ + 2][kSchurY + 2][kSchurX + 2], st[kSchurZ + 1][kSchurY + 1][kSchurX + 1];
    const int P = n + 1, t = int(threadIdx.x);
    const int i0 = int(blockIdx.x) * kSchurX, j0 = int(blockIdx.y) * kSchurY, k0 = int(blockIdx.z) * kSchurZ;
    for (int e = t; e < (kSchurX + 2) * (kSchurY + 2) * (kSchurZ + 2); e += kSchurX * kSchurY * kSchurZ) {
        const int i = e % (kSchurX + 2), j = (e / (kSchurX + 2)) % (kSchurY + 2), k = e / ((kSchurX + 2) * (kSchurY + 2));
        zt[k][j][i] = schur_z(n, z, i0 + i - 1, j0 + j - 1, k0 + k - 1);
    }
    for (int e = t; e < (kSchurX + 1) * (kSchurY + 1) * (kSchurZ + 1); e += kSchurX * kSchurY * kSchurZ) {
        const int i = e % (kSchurX + 1), j = (e / (kSchurX + 1)) % (kSchurY + 1), k = e / ((kSchurX + 1) * (kSchurY + 1));
        st[k][j][i] = schur_scale(n, scale, i0 + i - 1, j0 + j - 1, k0 + k - 1);
    }
    __syncthreads();
    const int x = t % kSchurX, y = (t / kSchurX) % kSchurY, w = t / (kSchurX * kSchurY);
    if (i0 + x >= P || j0 + y >= P || k0 + w >= P) return;
    const double mz = schur_sum([&](int i, int j, int k) { return zt[w + k][y + j][x + i]; },
                                [&](int i, int j, int k) { return st[w + k][y + j][x + i]; });
    schur_update(mz, r, dinv, z, d, z_new, d_new, c1, c2, size_t(i0 + x) + size_t(P) * ((j0 + y) + size_t(P) * (k0 + w)));
}

__global__ void k_mass_p_diag(int n, double h, const double* __restrict__ mu, double* __restrict__ diag,
                              double* __restrict__ weights) {
    const size_t vtx = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int P = n + 1;
    if (vtx >= size_t(P) * P * P) return;
    const int vi = int(vtx % P), vj = int((vtx / P) % P), vk = int(vtx / (size_t(P) * P));
    const double h3 = h * h * h;
    // int psi over one cell for a vertex: product of 1D sum_q w_q psi(q) = 1/2 each
    const double int1 = q2::gw(0) * q2::Pq(0, 0) + q2::gw(1) * q2::Pq(1, 0) + q2::gw(2) * q2::Pq(2, 0);
    const double mii = q2::M1(0, 0) * q2::M1(0, 0) * q2::M1(0, 0);
    double d = 0.0, wsum = 0.0;
    for (int dk = -1; dk <= 0; ++dk)
        for (int dj = -1; dj <= 0; ++dj)
            for (int di = -1; di <= 0; ++di) {
                const int ci = vi + di, cj = vj + dj, ck = vk + dk;
                if (ci < 0 || cj < 0 || ck < 0 || ci >= n || cj >= n || ck >= n) continue;
                const size_t cell = size_t(ci) + size_t(n) * (cj + size_t(n) * ck);
                d += h3 * mii / mu[cell];
                wsum += h3 * int1 * int1 * int1;
            }
    diag[vtx] = d;
    if (weights) weights[vtx] = wsum;
}

// ---------------------------------------------------------------- diagonal of A
__global__ void k_ref_diag(double* out81) {
    const int t = threadIdx.x;
    if (t >= 81) return;
    double u[3][27], w[3][27];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int a = 0; a < 27; ++a) u[c][a] = (c * 27 + a == t) ? 1.0 : 0.0;
    q2::cell_A(u, w);
    double v = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int a = 0; a < 27; ++a)
            if (c * 27 + a == t) v = w[c][a];
    out81[t] = v;
}

__global__ void k_inv_diag(int n, double h, const double* __restrict__ mu, const double* __restrict__ ref,
                           double* __restrict__ dinv) {
    const size_t node = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int M = 2 * n + 1;
    const size_t nodes = size_t(M) * M * M;
    if (node >= nodes) return;
    const int gi = int(node % M), gj = int((node / M) % M), gk = int(node / (size_t(M) * M));
    if (on_bnd(gi, M) || on_bnd(gj, M) || on_bnd(gk, M)) {
        for (int c = 0; c < 3; ++c) dinv[c * nodes + node] = 0.0;
        return;
    }
    // cells containing the node along one axis: odd index -> one cell (local 1); even -> two (local 2, 0)
    int cx[2], lx[2], nx = 0, cy[2], ly[2], ny = 0, cz[2], lz[2], nz = 0;
    auto axis = [n](int g, int* cc, int* ll, int& cnt) {
        if (g & 1) { cc[0] = (g - 1) / 2; ll[0] = 1; cnt = 1; return; }
        cnt = 0;
        if (g / 2 - 1 >= 0) { cc[cnt] = g / 2 - 1; ll[cnt] = 2; ++cnt; }
        if (g / 2 < n) { cc[cnt] = g / 2; ll[cnt] = 0; ++cnt; }
    };
    axis(gi, cx, lx, nx); axis(gj, cy, ly, ny); axis(gk, cz, lz, nz);
    double d[3] = {0.0, 0.0, 0.0};
    for (int c3 = 0; c3 < nz; ++c3)
        for (int c2 = 0; c2 < ny; ++c2)
            for (int c1 = 0; c1 < nx; ++c1) {
                const size_t cell = size_t(cx[c1]) + size_t(n) * (cy[c2] + size_t(n) * cz[c3]);
                const int a = lx[c1] + 3 * ly[c2] + 9 * lz[c3];
                const double s = mu[cell] * h;
                for (int c = 0; c < 3; ++c) d[c] += s * ref[c * 27 + a];
            }
    for (int c = 0; c < 3; ++c) dinv[c * nodes + node] = 1.0 / d[c];
}

// ---------------------------------------------------------------- sinker coefficients
__device__ __forceinline__ double sinker_X(double x, double y, double z, const double* __restrict__ centres, int ns,
                                           double delta, double omega) {
    double X = 1.0;
    for (int s = 0; s < ns; ++s) {
        const double dx = x - centres[3 * s], dy = y - centres[3 * s + 1], dz = z - centres[3 * s + 2];
        const double dist = sqrt(dx * dx + dy * dy + dz * dz);
        const double e = fmax(0.0, dist - 0.5 * omega);
        X *= 1.0 - exp(-delta * e * e);
    }
    return X;
}

__global__ void k_mu_sinker(int n, double h, const double* __restrict__ centres, int ns, double mu_min,
                            double mu_max, double delta, double omega, double* __restrict__ mu) {
    const size_t cell = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= size_t(n) * n * n) return;
    const int ci = int(cell % n), cj = int((cell / n) % n), ck = int(cell / (size_t(n) * n));
    double inv = 0.0, wsum = 0.0;
    for (int qz = 0; qz < 3; ++qz)
        for (int qy = 0; qy < 3; ++qy)
            for (int qx = 0; qx < 3; ++qx) {
                const double x = (ci + q2::gp(qx)) * h, y = (cj + q2::gp(qy)) * h, z = (ck + q2::gp(qz)) * h;
                const double X = sinker_X(x, y, z, centres, ns, delta, omega);
                const double m = X * mu_min + (1.0 - X) * mu_max;
                const double wq = q2::gw(qx) * q2::gw(qy) * q2::gw(qz);
                inv += wq / m;
                wsum += wq;
            }
    mu[cell] = wsum / inv;
}

__global__ void k_mu_from_q(size_t cells, const double* __restrict__ mu_q, double* __restrict__ mu) {
    const size_t cell = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= cells) return;
    double inv = 0.0, wsum = 0.0;
    for (int q = 0; q < 27; ++q) {
        const double wq = q2::gw(q % 3) * q2::gw((q / 3) % 3) * q2::gw(q / 9);
        inv += wq / mu_q[cell * 27 + q];
        wsum += wq;
    }
    mu[cell] = wsum / inv;
}

__global__ void k_mu_restrict(int nc, const double* __restrict__ fine, double* __restrict__ coarse) {
    const size_t cell = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= size_t(nc) * nc * nc) return;
    const int ci = int(cell % nc), cj = int((cell / nc) % nc), ck = int(cell / (size_t(nc) * nc));
    const int nf = 2 * nc;
    double s = 0.0;
    for (int k = 0; k < 2; ++k)
        for (int j = 0; j < 2; ++j)
            for (int i = 0; i < 2; ++i) s += fine[size_t(2 * ci + i) + size_t(nf) * (2 * cj + j + size_t(nf) * (2 * ck + k))];
    coarse[cell] = s / 8.0;
}

__global__ void k_rhs_sinker(int n, double h, const double* __restrict__ centres, int ns, double delta,
                             double omega, double beta, double* __restrict__ F) {
    const size_t cell = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (cell >= size_t(n) * n * n) return;
    const int ci = int(cell % n), cj = int((cell / n) % n), ck = int(cell / (size_t(n) * n));
    const int M = 2 * n + 1;
    const size_t nodes = size_t(M) * M * M;
    double f[27];
    for (int qz = 0; qz < 3; ++qz)
        for (int qy = 0; qy < 3; ++qy)
            for (int qx = 0; qx < 3; ++qx) {
                const double x = (ci + q2::gp(qx)) * h, y = (cj + q2::gp(qy)) * h, z = (ck + q2::gp(qz)) * h;
                const double X = sinker_X(x, y, z, centres, ns, delta, omega);
                f[qx + 3 * qy + 9 * qz] = q2::gw(qx) * q2::gw(qy) * q2::gw(qz) * beta * (X - 1.0);
            }
    q2::interpT<0>(f); q2::interpT<1>(f); q2::interpT<2>(f);
    const double h3 = h * h * h;
    for (int k = 0; k < 3; ++k)
        for (int j = 0; j < 3; ++j)
            for (int i = 0; i < 3; ++i) {
                const int gi = 2 * ci + i, gj = 2 * cj + j, gk = 2 * ck + k;
                if (on_bnd(gi, M) || on_bnd(gj, M) || on_bnd(gk, M)) continue;
                const size_t node = size_t(gi) + size_t(M) * (gj + size_t(M) * gk);
                atomicAdd(F + 2 * nodes + node, h3 * f[i + 3 * j + 9 * k]);
            }
}

inline unsigned blocks_for(size_t n, int t) { return unsigned((n + t - 1) / t); }

}  // namespace

template <typename T>
cudaError_t launch_copy_boundary(const LevelGeom& g, const T* in, T* out, cudaStream_t s) {
    const size_t nb = 6 * size_t(g.M) * g.M;
    LAUNCH(PROF_SMOOTH_VEC, s, k_copy_boundary<T><<<blocks_for(nb, 256), 256, 0, s>>>(g.M, in, out));
    return cudaGetLastError();
}
template cudaError_t launch_copy_boundary<float>(const LevelGeom&, const float*, float*, cudaStream_t);
template cudaError_t launch_copy_boundary<double>(const LevelGeom&, const double*, double*, cudaStream_t);

template <typename T>
cudaError_t launch_zero_boundary(const LevelGeom& g, T* x, cudaStream_t s) {
    return launch_copy_boundary<T>(g, nullptr, x, s);
}
template cudaError_t launch_zero_boundary<float>(const LevelGeom&, float*, cudaStream_t);
template cudaError_t launch_zero_boundary<double>(const LevelGeom&, double*, cudaStream_t);

template <typename T>
cudaError_t launch_free_rows(const LevelGeom& g, const T* x, const double* r, double* z, cudaStream_t s) {
    LAUNCH(PROF_CAST, s, (k_free_rows<T><<<blocks_for(g.nodes, 256), 256, 0, s>>>(g.M, x, r, z)));
    return cudaGetLastError();
}
template cudaError_t launch_free_rows<float>(const LevelGeom&, const float*, const double*, double*, cudaStream_t);
template cudaError_t launch_free_rows<double>(const LevelGeom&, const double*, const double*, double*, cudaStream_t);

cudaError_t launch_stokes_blocks(const LevelGeom& g, const double* mu, const double* src_u, const double* src_p,
                                 double* dst_u, double* dst_p, bool do_a, bool do_bt, bool do_b, cudaStream_t s) {
    cudaError_t e;
    if (!do_a && do_bt && !do_b) {   // B^T alone: the gather, and the boundary rows
        LAUNCH(PROF_BT_F64, s, (k_bt<BT_PLAIN, double, false><<<blocks_for(g.cells, 128), 128, 0, s>>>(g.n, g.h, src_p, nullptr, dst_u)));
        return launch_zero_boundary<double>(g, dst_u, s);
    }
    if (do_a || do_bt) {
        e = cudaMemsetAsync(dst_u, 0, g.n_u * sizeof(double), s);
        if (e != cudaSuccess) return e;
    }
    if (do_b) {
        e = cudaMemsetAsync(dst_p, 0, g.n_p * sizeof(double), s);
        if (e != cudaSuccess) return e;
    }
    e = launch_outer_fix(g, mu, src_u, src_p, dst_u, dst_p, do_a, do_bt, do_b, s);
    if (e != cudaSuccess) return e;
    if (do_a) {
        const size_t nbd = 6 * size_t(g.M) * g.M;
        LAUNCH(PROF_SMOOTH_VEC, s, (k_copy_boundary<double><<<blocks_for(nbd, 256), 256, 0, s>>>(g.M, src_u, dst_u)));
    }
    return cudaGetLastError();
}

cudaError_t launch_mass_p(const LevelGeom& g, const double* mu, const double* src, double* dst, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(dst, 0, g.n_p * sizeof(double), s);
    if (e != cudaSuccess) return e;
    LAUNCH(PROF_MASS_P, s, k_mass_p<<<blocks_for(g.cells, 128), 128, 0, s>>>(g.n, g.h, mu, src, dst));
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_bt_resid(const LevelGeom& g, const double* p, const double* r, T* out, bool df, cudaStream_t s) {
    if (sizeof(T) == 4 && df)
        LAUNCH(PROF_BT_F64, s, (k_bt<BT_RESID, T, sizeof(T) == 4><<<blocks_for(g.cells, 128), 128, 0, s>>>(g.n, g.h, p, r, out)));
    else
        LAUNCH(PROF_BT_F64, s, (k_bt<BT_RESID, T, false><<<blocks_for(g.cells, 128), 128, 0, s>>>(g.n, g.h, p, r, out)));
    return cudaGetLastError();
}
template cudaError_t launch_bt_resid<float>(const LevelGeom&, const double*, const double*, float*, bool, cudaStream_t);
template cudaError_t launch_bt_resid<double>(const LevelGeom&, const double*, const double*, double*, bool, cudaStream_t);

cudaError_t launch_mass_scale(const LevelGeom& g, const double* mu, double* scale, cudaStream_t s) {
    LAUNCH(PROF_MASS_P, s, k_mass_scale<<<blocks_for(g.cells, 256), 256, 0, s>>>(g.cells, g.h, mu, scale));
    return cudaGetLastError();
}

cudaError_t launch_schur_cheb(const LevelGeom& g, const double* scale, const double* r, const double* dinv,
                              const double* z, const double* d, double* z_new, double* d_new, double c1, double c2,
                              cudaStream_t s) {
    const unsigned P = unsigned(g.n) + 1;
    const dim3 grid((P + kSchurX - 1) / kSchurX, (P + kSchurY - 1) / kSchurY, (P + kSchurZ - 1) / kSchurZ);
    LAUNCH(PROF_MASS_P, s, (k_schur_cheb<<<grid, kSchurX * kSchurY * kSchurZ, 0, s>>>(g.n, scale, r, dinv, z, d, z_new, d_new, c1, c2)));
    return cudaGetLastError();
}

cudaError_t launch_mass_p_diag(const LevelGeom& g, const double* mu, double* diag, double* weights,
                               cudaStream_t s) {
    LAUNCH(PROF_SMOOTH_VEC, s, k_mass_p_diag<<<blocks_for(g.n_p, 256), 256, 0, s>>>(g.n, g.h, mu, diag, weights));
    return cudaGetLastError();
}

cudaError_t launch_ref_diag(double* ref_diag81, cudaStream_t s) {
    LAUNCH(PROF_SMOOTH_VEC, s, k_ref_diag<<<1, 96, 0, s>>>(ref_diag81));
    return cudaGetLastError();
}

cudaError_t launch_inv_diag(const LevelGeom& g, const double* mu, const double* ref_diag81, double* dinv,
                            cudaStream_t s) {
    LAUNCH(PROF_SMOOTH_VEC, s, k_inv_diag<<<blocks_for(g.nodes, 256), 256, 0, s>>>(g.n, g.h, mu, ref_diag81, dinv));
    return cudaGetLastError();
}

cudaError_t launch_mu_sinker(const LevelGeom& g, const double* centres, int n_sinkers, double mu_min,
                             double mu_max, double delta, double omega, double* mu, cudaStream_t s) {
    LAUNCH(PROF_SMOOTH_VEC, s, k_mu_sinker<<<blocks_for(g.cells, 128), 128, 0, s>>>(g.n, g.h, centres, n_sinkers, mu_min, mu_max, delta,
                                                          omega, mu));
    return cudaGetLastError();
}

cudaError_t launch_mu_from_q(const LevelGeom& g, const double* mu_q, double* mu, cudaStream_t s) {
    LAUNCH(PROF_SMOOTH_VEC, s, k_mu_from_q<<<blocks_for(g.cells, 128), 128, 0, s>>>(g.cells, mu_q, mu));
    return cudaGetLastError();
}

cudaError_t launch_mu_restrict(const LevelGeom& coarse, const double* mu_fine, double* mu_coarse, cudaStream_t s) {
    LAUNCH(PROF_SMOOTH_VEC, s, k_mu_restrict<<<blocks_for(coarse.cells, 128), 128, 0, s>>>(coarse.n, mu_fine, mu_coarse));
    return cudaGetLastError();
}

cudaError_t launch_rhs_sinker(const LevelGeom& g, const double* centres, int n_sinkers, double delta,
                              double omega, double beta, double* F, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(F, 0, g.n_u * sizeof(double), s);
    if (e != cudaSuccess) return e;
    LAUNCH(PROF_SMOOTH_VEC, s, k_rhs_sinker<<<blocks_for(g.cells, 128), 128, 0, s>>>(g.n, g.h, centres, n_sinkers, delta, omega, beta, F));
    return cudaGetLastError();
}

}  // namespace stk
