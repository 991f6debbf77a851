// pressure.cuh -- per-thread bodies of the pressure-side gathers of the preconditioner on uniform
// meshes (ops.cu kernels k_bt and k_schur_cheb): B^T p as a tensor product of assembled 1D
// moment operators (Section 2.1, definition of B), and one Jacobi-Chebyshev step of S_hat^-1 on
// the 1/mu-weighted pressure mass matrix (Section 2.2.2) with M_p gathered per vertex, its
// products in double-float on the FP32 pipes. Plain functions of the thread's indices, so
// that a host program can run them node by node and vertex by vertex.
#pragma once

#include "df64.cuh"
#include "q2_basis.cuh"

namespace stk {

// ---- B^T. B^T carries no viscosity, so component c of B^T p is -h^2 (X_2 x X_1 x X_0) p with X_d
// the 1D moment operator assembled over the cells along axis d (DP, the moments of the Q2 basis
// derivatives against the Q1 basis, along axis c; VP, those of the basis itself, along the other
// two). An interior Q2 node 2e (a vertex) has the row (XP(2,0), XP(2,1) + XP(0,0), XP(0,1)) at
// vertices e-1, e, e+1, an interior node 2e+1 the row (XP(1,0), XP(1,1)) at e, e+1. For the line
// (J, K) of component C: t_e = sum X_1[J][b] X_2[K][k] p(e, b, k), then the x-nodes 2e and 2e+1
// from t_{e-1}, t_e, t_{e+1}; boundary nodes get 0, as in the cell kernels.

// Evaluated, the rows are (1, 0, -1)/6 and (4, -4)/6 along axis c and (0, 2, 0)/6 and (2, 2)/6 along the
// others: sums and differences of neighbouring vertices, one factor per node. bt_nodes forms the 8 nodes
// (2e, 2e + 1) x (2f, 2f + 1) x (2g, 2g + 1) of component C from the 3 x 3 x 3 vertices around (e, f, g)
// (v[k][j][i] at e - 1 + i, ...; nodes with an even index 0 are boundary nodes, whatever v holds
// there): out[i + 2 j + 4 k] without the factor -h^2 bt_factor. 16 additions for 8 nodes.
template <int C>
__host__ __device__ constexpr double bt_factor(int i, int j, int k) {   // i, j, k: node parity (1: odd)
    return ((C == 0 ? i : (C == 1 ? j : k)) != 0 ? 2.0 / 3.0 : 1.0 / 6.0) / 9.0;
}
template <int C, typename T>
__host__ __device__ __forceinline__ void bt_nodes(const T (&v)[3][3][3], T (&out)[8]) {
    auto at = [&v](int d, int a, int b) -> const T& {   // d along C, then the other two axes in order
        return C == 0 ? v[1 + b][1 + a][1 + d] : (C == 1 ? v[1 + b][1 + d][1 + a] : v[1 + d][1 + b][1 + a]);
    };
    T x[2][2][2];   // [parity along C][a][b]
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            x[0][a][b] = at(-1, a, b) - at(1, a, b);
            x[1][a][b] = at(0, a, b) - at(1, a, b);
        }
#pragma unroll
    for (int d = 0; d < 2; ++d) {
#pragma unroll
        for (int b = 0; b < 2; ++b) x[d][1][b] = x[d][0][b] + x[d][1][b];   // now parity along a
#pragma unroll
        for (int a = 0; a < 2; ++a) x[d][a][1] = x[d][a][0] + x[d][a][1];   // and along b
    }
#pragma unroll
    for (int d = 0; d < 2; ++d)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const int i = C == 0 ? d : a, j = C == 0 ? a : (C == 1 ? d : b), k = C == 2 ? d : b;
                out[i + 2 * j + 4 * k] = x[d][a][b];
            }
}

// The same per x-line of nodes, with the moments as weights in double-float (host comparison).
// entry of X_0 (axis 0) in row i at vertex a, for the rows of vertex e (i = 2e, 2e + 1)
template <int C>
__host__ __device__ __forceinline__ double bt_x_row(int i, int a, int e) {
    constexpr bool D = C == 0;
    auto xp = [](int m, int v) { return D ? q2::DP(m, v) : q2::VP(m, v); };
    if (i & 1) return a == e ? xp(1, 0) : (a == e + 1 ? xp(1, 1) : 0.0);
    return a == e - 1 ? xp(2, 0) : (a == e ? xp(2, 1) + xp(0, 0) : (a == e + 1 ? xp(0, 1) : 0.0));
}

// row i of X_AX (interior i) over the vertices i/2 - 1, i/2, i/2 + 1
template <int C, int AX>
__host__ __device__ __forceinline__ void bt_row(int i, double (&w)[3]) {
    constexpr bool D = C == AX;
    auto xp = [](int m, int v) { return D ? q2::DP(m, v) : q2::VP(m, v); };
    if (i & 1) {   // vertices i/2, i/2 + 1
        w[0] = 0.0;
        w[1] = xp(1, 0);
        w[2] = xp(1, 1);
    } else {
        w[0] = xp(2, 0);
        w[1] = xp(2, 1) + xp(0, 0);
        w[2] = xp(0, 1);
    }
}

// weight q (= b-slot + 3 k-slot) of the interior line (J, K)
template <int C>
__host__ __device__ __forceinline__ q2::df64 bt_weight(int J, int K, int q) {
    double wy[3], wz[3];
    bt_row<C, 1>(J, wy);
    bt_row<C, 2>(K, wz);
    return q2::split_double(wy[q % 3] * wz[q / 3]);
}

// t_e of the interior line (J, K) from the line's 9 weights w
template <int C>
__host__ __device__ __forceinline__ q2::df64 bt_t(int n, const double* __restrict__ p, int J, int K, int e,
                                                   const q2::df64* w) {
    const int P = n + 1;
    const int by = J / 2 - 1, bz = K / 2 - 1;
    q2::df64 acc;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const int b = by + q % 3, k = bz + q / 3;
        if (b < 0 || b >= P || k < 0 || k >= P) continue;   // zero weights only
        q2::mac(acc, w[q], q2::split_double(p[size_t(e) + size_t(P) * (b + size_t(P) * k)]));
    }
    q2::renorm(acc);
    return acc;
}

// the x-nodes 2e and 2e + 1 (e < n) of the interior line whose first node is o, times s = -h^2
template <int C>
__host__ __device__ __forceinline__ void bt_out(int n, double s, double* __restrict__ o, int e, const q2::df64* t) {
    using q2::df64;
    const int M = 2 * n + 1;
    const int i0 = 2 * e;
    if (i0 == 0 || i0 == M - 1) {
        o[i0] = 0.0;
    } else {
        df64 v;
        q2::mac(v, df64(bt_x_row<C>(i0, e - 1, e)), t[e - 1]);
        q2::mac(v, df64(bt_x_row<C>(i0, e, e)), t[e]);
        q2::mac(v, df64(bt_x_row<C>(i0, e + 1, e)), t[e + 1]);
        q2::renorm(v);
        o[i0] = s * v.to_double();
    }
    if (e < n) {
        df64 v;
        q2::mac(v, df64(bt_x_row<C>(i0 + 1, e, e)), t[e]);
        q2::mac(v, df64(bt_x_row<C>(i0 + 1, e + 1, e)), t[e + 1]);
        q2::renorm(v);
        o[i0 + 1] = s * v.to_double();
    }
}

// ---- S_hat^-1 step at pressure vertex vtx:
//   d' = c1 d + c2 D^-1 (r - M_p z),  z' = z + d'   (into the other buffers of the pairs).
// (M_p z)_v sums the element products of the up to 8 cells around v, s_K sum_w m(v, w) z_w with
// s_K = h^3 / mu_K and m = M1 x M1 x M1, M1 = (2, 1; 1, 2)/6 on [0,1]: the sums of the 8 cells are formed
// together axis by axis (2 z_v + z_w towards each side: 38 additions for 64 products), the factor
// 1/216 at the end. In double-float: in FP64 the additions would bind the kernel to the FP64 pipe.
// z(i, j, k) is the vertex value at offset i - 1, j - 1, k - 1 from v, scale(i, j, k) the s_K of the cell towards
// side i, j, k (0: lower), 0 outside the mesh.
template <typename Z, typename S>
__host__ __device__ __forceinline__ double schur_sum(const Z& z, const S& scale) {
    using q2::df64;
    auto side = [](const df64& own, const df64& other) { return df64(own.hi + own.hi, own.lo + own.lo) + other; };
    df64 c[3][2][2];   // [k][side along y][side along x]
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        df64 a[3][2];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const df64 own = z(1, j, k);
            a[j][0] = side(own, z(0, j, k));
            a[j][1] = side(own, z(2, j, k));
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            c[k][0][i] = side(a[1][i], a[0][i]);
            c[k][1][i] = side(a[1][i], a[2][i]);
        }
    }
    df64 acc;
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) acc = acc + scale(i, j, k) * side(c[1][j][i], c[2 * k][j][i]);
    return acc.to_double() * (1.0 / 216.0);
}
__host__ __device__ __forceinline__ void schur_update(double mz, const double* __restrict__ r, const double* __restrict__ dinv,
                                                      const double* __restrict__ z, const double* __restrict__ d,
                                                      double* __restrict__ z_new, double* __restrict__ d_new, double c1,
                                                      double c2, size_t vtx) {
    const double dn = (c1 != 0.0 ? c1 * d[vtx] : 0.0) + c2 * (dinv[vtx] * (r[vtx] - mz));
    d_new[vtx] = dn;
    z_new[vtx] = z[vtx] + dn;
}
// The values that the step at one vertex needs, in double-float, 0 outside the mesh.
__host__ __device__ __forceinline__ q2::df64 schur_z(int n, const double* __restrict__ z, int i, int j, int k) {
    const int P = n + 1;
    return i >= 0 && j >= 0 && k >= 0 && i < P && j < P && k < P ? q2::split_double(z[size_t(i) + size_t(P) * (j + size_t(P) * k)])
                                                                 : q2::df64();
}
__host__ __device__ __forceinline__ q2::df64 schur_scale(int n, const double* __restrict__ scale, int i, int j, int k) {
    return i >= 0 && j >= 0 && k >= 0 && i < n && j < n && k < n ? q2::split_double(scale[size_t(i) + size_t(n) * (j + size_t(n) * k)])
                                                                 : q2::df64();
}
// One vertex on its own (k_schur_cheb runs the same with the values of a tile in shared memory).
__host__ __device__ __forceinline__ void schur_vertex(int n, const double* __restrict__ scale,
                                                      const double* __restrict__ r, const double* __restrict__ dinv,
                                                      const double* __restrict__ z, const double* __restrict__ d,
                                                      double* __restrict__ z_new, double* __restrict__ d_new,
                                                      double c1, double c2, size_t vtx) {
    const int P = n + 1;
    const int vi = int(vtx % P), vj = int((vtx / P) % P), vk = int(vtx / (size_t(P) * P));
    const double mz = schur_sum([&](int i, int j, int k) { return schur_z(n, z, vi + i - 1, vj + j - 1, vk + k - 1); },
                                [&](int i, int j, int k) { return schur_scale(n, scale, vi + i - 1, vj + j - 1, vk + k - 1); });
    schur_update(mz, r, dinv, z, d, z_new, d_new, c1, c2, vtx);
}

}  // namespace stk
