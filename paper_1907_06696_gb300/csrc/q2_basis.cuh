// q2_basis.cuh -- reference-cell tables and the sum-factorised cell kernels
// of the Q2-Q1 Stokes operators (Section 2.1, definitions of A, B, B^T, F;
// Section 2.2.2, weighted pressure mass matrix).
//
// Reference cell [0,1]^3. Q2 node (i,j,k) at (i/2, j/2, k/2), local index
// i + 3j + 9k. Gauss point (qx,qy,qz) of the 3-point Gauss-Legendre rule,
// local index qx + 3qy + 9qz. Q1 vertex (i,j,k) in {0,1}^3, index i + 2j + 4k.
//
// The velocity operator of one cube cell of side h with cell viscosity mu is
//   (A u)_(a,c) = mu h sum_q w_q sum_d sigma_cd(q) d_d phi_a(q),
//   sigma = grad_ref u + grad_ref u^T   (= 2 eps in reference coordinates),
// which on a cube is a fixed 81 x 81 matrix times mu h, a sum of tensor products
// of 1D integrals. It is applied in the Legendre modes of each axis, where those
// integrals are diagonal or have two entries (below): 1D transforms of the nodal
// values to the modes, a diagonal and a few products, and the transposed
// transforms. Every table is a compile-time constant and every loop fully
// unrolled, so each coefficient is an immediate operand of one FMA.
#pragma once

#include <cuda_runtime.h>

#include "df64.cuh"

namespace q2 {

// ---------------------------------------------------------------- constants
__host__ __device__ constexpr double csqrt_newton(double x, double g, int it) {
    return it == 0 ? g : csqrt_newton(x, 0.5 * (g + x / g), it - 1);
}
__host__ __device__ constexpr double csqrt(double x) { return csqrt_newton(x, x > 1.0 ? x : 1.0, 64); }

// 3-point Gauss-Legendre on [0,1]: 1/2 -+ sqrt(15)/10, 1/2; weights 5/18, 8/18, 5/18.
__host__ __device__ constexpr double goff() { return csqrt(15.0) / 10.0; }
__host__ __device__ constexpr double gp(int q) { return q == 0 ? 0.5 - goff() : (q == 1 ? 0.5 : 0.5 + goff()); }
__host__ __device__ constexpr double gw(int q) { return q == 1 ? 8.0 / 18.0 : 5.0 / 18.0; }

// Quadratic Lagrange basis on {0, 1/2, 1} and its derivative.
__host__ __device__ constexpr double lag(int m, double x) {
    return m == 0 ? (2.0 * x - 1.0) * (x - 1.0) : (m == 1 ? 4.0 * x * (1.0 - x) : x * (2.0 * x - 1.0));
}
__host__ __device__ constexpr double dlag(int m, double x) {
    return m == 0 ? 4.0 * x - 3.0 : (m == 1 ? 4.0 - 8.0 * x : 4.0 * x - 1.0);
}
// V[q][m] = l_m(g_q): nodal values -> Gauss-point values.
__host__ __device__ constexpr double Vq(int q, int m) { return lag(m, gp(q)); }
// Q1 basis on [0,1] at Gauss point q.
__host__ __device__ constexpr double Pq(int q, int v) { return v == 0 ? 1.0 - gp(q) : gp(q); }
// 1D Q1 mass matrix on [0,1] by the same quadrature.
__host__ __device__ constexpr double M1(int a, int b) {
    return gw(0) * Pq(0, a) * Pq(0, b) + gw(1) * Pq(1, a) * Pq(1, b) + gw(2) * Pq(2, a) * Pq(2, b);
}

// Linear index of (axis index a, other indices o1 < o2 in axis order).
template <int AX>
__host__ __device__ constexpr int lin(int a, int o1, int o2) {
    return AX == 0 ? a + 3 * o1 + 9 * o2 : (AX == 1 ? o1 + 3 * a + 9 * o2 : o1 + 3 * o2 + 9 * a);
}

// ---------------------------------------------------------------- 1D sweeps
// x <- V^T x along AX, in place (Gauss-point sums -> nodes).
template <int AX, typename T>
__host__ __device__ __forceinline__ void interpT(T* x) {
#pragma unroll
    for (int o2 = 0; o2 < 3; ++o2)
#pragma unroll
        for (int o1 = 0; o1 < 3; ++o1) {
            const T a0 = x[lin<AX>(0, o1, o2)], a1 = x[lin<AX>(1, o1, o2)], a2 = x[lin<AX>(2, o1, o2)];
#pragma unroll
            for (int m = 0; m < 3; ++m)
                x[lin<AX>(m, o1, o2)] = T(Vq(0, m)) * a0 + T(Vq(1, m)) * a1 + T(Vq(2, m)) * a2;
        }
}

// ---------------------------------------------------------------- Legendre modes
// A quadratic on [0,1] with nodal values a0, a1, a2 is w/6 P_0 + d/2 P_1 + e/3 P_2 in the Legendre
// polynomials of [0,1], with w = a0 + 4 a1 + a2, d = a2 - a0, e = a0 - 2 a1 + a2: small integers only.
// In these modes the 1D forms of the element integrals are diagonal or have two entries,
//   int u v   = w w'/36 + d d'/12 + e e'/45,   int u' v' = d d' + 4/3 e e',
//   int u v'  = w d'/6 + d e'/3,
// so the element operator is a diagonal plus 12 products per pair of components, and its cost is
// that of the transforms (4 operations a line each way): about 880 operations per cell against 2,633
// for sweeps through the Gauss points, with half their rounding error (the first and second
// differences of the nodal values are formed directly). One FP32 cell per thread with atomic adds took 320 us
// through the Gauss points at 128^3 and 229 us in the modes, at 64^3 50 and 37 us.
enum Mode { MODE_W = 0, MODE_D = 1, MODE_E = 2 };
__host__ __device__ constexpr double mode_mass(int a) { return a == 0 ? 1.0 / 36.0 : (a == 1 ? 1.0 / 12.0 : 1.0 / 45.0); }
__host__ __device__ constexpr double mode_stiff(int a) { return a == 0 ? 0.0 : (a == 1 ? 1.0 : 4.0 / 3.0); }
// int u v' couples mode a of u with mode a + 1 of v (a = 0, 1).
__host__ __device__ constexpr double mode_grad(int a) { return a == 0 ? 1.0 / 6.0 : 1.0 / 3.0; }
// Diagonal of row component c: 2 int d_c u d_c v + sum over the other axes of int d_d u d_d v.
__host__ __device__ constexpr double mode_diag(int c, int i, int j, int k) {
    return (c == 0 ? 2.0 : 1.0) * mode_stiff(i) * mode_mass(j) * mode_mass(k) +
           (c == 1 ? 2.0 : 1.0) * mode_mass(i) * mode_stiff(j) * mode_mass(k) +
           (c == 2 ? 2.0 : 1.0) * mode_mass(i) * mode_mass(j) * mode_stiff(k);
}

// Nodal values <-> modes along AX, in place: to_modes x <- (w, d, e), from_modes its transpose, which
// takes e twice (rows of the tables carry the factor 2 per index E, mode_out: w + e/2 and 4 w - e are
// one multiply-add each).
template <int AX, typename T>
__host__ __device__ __forceinline__ void to_modes(T* x) {
#pragma unroll
    for (int o2 = 0; o2 < 3; ++o2)
#pragma unroll
        for (int o1 = 0; o1 < 3; ++o1) {
            const T a0 = x[lin<AX>(0, o1, o2)], a1 = x[lin<AX>(1, o1, o2)], a2 = x[lin<AX>(2, o1, o2)];
            const T s = a0 + a2;
            x[lin<AX>(MODE_W, o1, o2)] = s + T(4) * a1;
            x[lin<AX>(MODE_D, o1, o2)] = a2 - a0;
            x[lin<AX>(MODE_E, o1, o2)] = s - T(2) * a1;
        }
}
template <int AX, typename T>
__host__ __device__ __forceinline__ void from_modes(T* x) {
#pragma unroll
    for (int o2 = 0; o2 < 3; ++o2)
#pragma unroll
        for (int o1 = 0; o1 < 3; ++o1) {
            const T w = x[lin<AX>(MODE_W, o1, o2)], d = x[lin<AX>(MODE_D, o1, o2)], e = x[lin<AX>(MODE_E, o1, o2)];
            const T t = w + T(0.5) * e;
            x[lin<AX>(0, o1, o2)] = t - d;
            x[lin<AX>(1, o1, o2)] = T(4) * w - e;
            x[lin<AX>(2, o1, o2)] = t + d;
        }
}
template <typename T>
__host__ __device__ __forceinline__ void to_modes3(T* x) { to_modes<0>(x); to_modes<1>(x); to_modes<2>(x); }
template <typename T>
__host__ __device__ __forceinline__ void from_modes3(T* x) { from_modes<2>(x); from_modes<1>(x); from_modes<0>(x); }

__host__ __device__ constexpr double mode_out(int i, int j, int k) {
    return (i == 2 ? 2.0 : 1.0) * (j == 2 ? 2.0 : 1.0) * (k == 2 ? 2.0 : 1.0);
}

// Contribution of column component D to mode (i,j,k) of row component C (C != D):
// int d_C u_D d_D v_C couples v's mode a along C with u's a + 1, and v's b along D with u's b - 1.
template <int C, int D>
__host__ __device__ constexpr int mode_partner(int i, int j, int k) {
    const int m[3] = {i, j, k};
    if (m[C] > 1 || m[D] < 1) return -1;
    const int b0 = i + (C == 0) - (D == 0), b1 = j + (C == 1) - (D == 1), b2 = k + (C == 2) - (D == 2);
    return b0 + 3 * b1 + 9 * b2;
}
template <int C, int D>
__host__ __device__ constexpr double mode_cross(int i, int j, int k) {
    const int m[3] = {i, j, k};
    return mode_grad(m[C]) * mode_grad(m[D] - 1) * mode_mass(m[3 - C - D]);
}

// Modes of row component C of the velocity operator (times mode_out): w = (A U)_C without mu h, U1 and U2
// the modes of components (C + 1) % 3 and (C + 2) % 3.
template <int C, typename T>
__host__ __device__ __forceinline__ void modes_A(const T* U, const T* U1, const T* U2, T* w) {
    constexpr int D1 = (C + 1) % 3, D2 = (C + 2) % 3;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int m = i + 3 * j + 9 * k;
                T v = T(0);
                if (m != 0) v = T(mode_diag(C, i, j, k) * mode_out(i, j, k)) * U[m];
                const int p1 = mode_partner<C, D1>(i, j, k), p2 = mode_partner<C, D2>(i, j, k);
                if (p1 >= 0) v += T(mode_cross<C, D1>(i, j, k) * mode_out(i, j, k)) * U1[p1 < 0 ? 0 : p1];
                if (p2 >= 0) v += T(mode_cross<C, D2>(i, j, k) * mode_out(i, j, k)) * U2[p2 < 0 ? 0 : p2];
                w[m] = v;
            }
}

// ---------------------------------------------------------------- cell kernels
// Velocity operator of one reference cell, without the factor mu h:
// in: u[c][a] nodal values (overwritten by their modes);
// out: w[c][a] = int sum_d sigma_cd d_d phi_a, sigma = grad u + grad u^T.
template <typename T>
__host__ __device__ __forceinline__ void cell_A(T (&u)[3][27], T (&w)[3][27]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) to_modes3(u[c]);
    modes_A<0>(u[0], u[1], u[2], w[0]);
    modes_A<1>(u[1], u[2], u[0], w[1]);
    modes_A<2>(u[2], u[0], u[1], w[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) from_modes3(w[c]);
}

// ---- B and B^T in the modes: a Q1 pressure with vertex values p0, p1 along an axis has the modes
// P = p0 + p1, D = p1 - p0 (p = P/2 + D/2 P_1), and int v p = (w P + d D)/12, int v' p = d P/2 + e D/3.
// So mode (i,j,k) of component C meets the pressure mode with index i - 1 along C and i elsewhere (outer.cuh).
// Vertex values -> pressure modes (in place), and the transpose.
template <typename T>
__host__ __device__ __forceinline__ void to_pressure_modes(T (&p)[8]) {
#pragma unroll
    for (int s = 1; s < 8; s *= 2)
#pragma unroll
        for (int v = 0; v < 8; ++v)
            if (!(v & s)) {
                const T a = p[v], b = p[v + s];
                p[v] = a + b;
                p[v + s] = b - a;
            }
}
template <typename T>
__host__ __device__ __forceinline__ void from_pressure_modes(T (&p)[8]) {
#pragma unroll
    for (int s = 1; s < 8; s *= 2)
#pragma unroll
        for (int v = 0; v < 8; ++v)
            if (!(v & s)) {
                const T a = p[v], b = p[v + s];
                p[v] = a - b;
                p[v + s] = a + b;
            }
}
// 1D moments of the Q2 basis against the Q1 basis on [0,1], exact by the same
// quadrature: VP(m,v) = int l_m psi_v, DP(m,v) = int l_m' psi_v.
__host__ __device__ constexpr double VP(int m, int v) {
    return gw(0) * lag(m, gp(0)) * Pq(0, v) + gw(1) * lag(m, gp(1)) * Pq(1, v) + gw(2) * lag(m, gp(2)) * Pq(2, v);
}
__host__ __device__ constexpr double DP(int m, int v) {
    return gw(0) * dlag(m, gp(0)) * Pq(0, v) + gw(1) * dlag(m, gp(1)) * Pq(1, v) + gw(2) * dlag(m, gp(2)) * Pq(2, v);
}
// 1D factor of int d_c(phi_m) psi_v along axis AX for velocity component C.
template <int C, int AX>
__host__ __device__ constexpr double XP(int m, int v) { return C == AX ? DP(m, v) : VP(m, v); }

// out_c(i,j,k) (+)= sum_v [int d_c(phi_ijk) psi_v] p_v on the reference cell: the
// tensor product of three 3x2 moment matrices, applied axis by axis (B^T without h).
template <int C, typename T>
__host__ __device__ __forceinline__ void bt_component(const T (&p)[8], T* out) {
    T s1[3][2][2], s2[3][3][2];
#pragma unroll
    for (int d = 0; d < 2; ++d)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int i = 0; i < 3; ++i)
                s1[i][b][d] = T(XP<C, 0>(i, 0)) * p[0 + 2 * b + 4 * d] + T(XP<C, 0>(i, 1)) * p[1 + 2 * b + 4 * d];
#pragma unroll
    for (int d = 0; d < 2; ++d)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i)
                s2[i][j][d] = T(XP<C, 1>(j, 0)) * s1[i][0][d] + T(XP<C, 1>(j, 1)) * s1[i][1][d];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i)
                out[i + 3 * j + 9 * k] += T(XP<C, 2>(k, 0)) * s2[i][j][0] + T(XP<C, 2>(k, 1)) * s2[i][j][1];
}

// out_v += sum_(c,m) [int d_c(phi_m) psi_v] u_c(m): the transpose (B without h).
template <int C, typename T>
__host__ __device__ __forceinline__ void b_component(const T* u, T (&out)[8]) {
    T t1[3][3][2], t2[3][2][2];
#pragma unroll
    for (int d = 0; d < 2; ++d)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i)
                t1[i][j][d] = T(XP<C, 2>(0, d)) * u[i + 3 * j] + T(XP<C, 2>(1, d)) * u[i + 3 * j + 9] +
                              T(XP<C, 2>(2, d)) * u[i + 3 * j + 18];
#pragma unroll
    for (int d = 0; d < 2; ++d)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int i = 0; i < 3; ++i)
                t2[i][b][d] = T(XP<C, 1>(0, b)) * t1[i][0][d] + T(XP<C, 1>(1, b)) * t1[i][1][d] +
                              T(XP<C, 1>(2, b)) * t1[i][2][d];
#pragma unroll
    for (int d = 0; d < 2; ++d)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int a = 0; a < 2; ++a)
                out[a + 2 * b + 4 * d] += T(XP<C, 0>(0, a)) * t2[0][b][d] + T(XP<C, 0>(1, a)) * t2[1][b][d] +
                                          T(XP<C, 0>(2, a)) * t2[2][b][d];
}

}  // namespace q2
