// outer.cuh -- the FP64-interface outer Stokes blocks [A, B^T; B, 0]
// (Section 2.1, eq. stokes_linear_system) in fixed point, in the Legendre modes of
// q2_basis.cuh, with one velocity component per thread.
//
// GB300 issues one FP64 instruction per ~38 integer ones, and the transforms between nodal values
// and modes multiply by 1, 2 and 4 only. So each cell's values are written once as 64-bit integers
// against the cell's largest magnitude and everything up to the last scaling is integer arithmetic,
// exact but for the bits it drops:
//   u = X 2^(Eu - 54), |X| <= 2^54 (rounding 2^-55 of the cell's largest |u|), modes
//       U = (T x T x T) X, |U| <= 2^(54 + 7.76);
//   97200 A is an integer matrix in the modes (stiffness (0,3,4)/3, mass (5,15,4)/180, derivative
//       couplings (1,2)/6): Y = 97200 A U, |Y| <= 2^(54 + 15.99), formed in 96 bits and kept without
//       its lowest 12;
//   B^T p is added as (3|2) p' with p' = 112.5 h/mu p in the same units (fix_factor);
//   the transposed transform gives |result| < 2^(42 + 20.43) (sums that leave 64 bits on the way
//       return: two's complement), rounded to 53 bits and multiplied by mu h 2^E / 97200.
// B u is (3|2) U / 864 without its lowest 2 bits, |result| <= 2^(52 + 10.1).
// The error is that of FP64 arithmetic (measured against exact sums on 12^3 cells, velocity rows: 1.2e-16
// relative on random and 2.7e-16 on smooth fields; sum factorisation in FP64 4.8e-16 and 2.3e-15,
// in double-float pairs 6.4e-15 and 3.6e-14), against the size of the cell's values: a value far below its
// cell's largest keeps the bits above 2^-55 of that one. With nodal values over 8 decades at random within every cell
// (4^3) the error is 1.6e-16 in the 2-norm and 4e-14 of (|A| |u|) in the worst row; sum factorisation in FP64, which mixes a
// cell's values too, 3.2e-16 and 1.5e-14. Where B^T p is the larger term (|p| 1e4 and 1e6, 3^3 to 8^3 cells) 1.5e-16 to
// 2.6e-16 in the 2-norm; in FP64 2.1e-16 to 2.8e-16. On octrees of 4,635 and 15,548 leaves (viscosity ratio 1e6, against
// sums in extended precision) 1.8e-16; in FP64 3.7e-16.
//
// A CTA holds 32 cells and 96 threads; warp c owns velocity component c of
// the 32 cells (lane g = cell g) and the three exchange their modes through shared memory (20.7 KB).
// The phases are plain functions of the thread index so that a host program
// can run them and compare with the oracle.
#pragma once

#include <cstring>

#include "df64.cuh"
#include "q2_basis.cuh"

namespace stk {

constexpr int kOuterCells = 32;       // cells per CTA
constexpr int kOuterThreads = 96;     // 3 components x 32 cells

struct OuterArgs {
    int n, M;
    size_t nodes;
    double h;
    const double* mu;
    const double* src_u;
    const double* src_p;
    double* dst_u;
    double* dst_p;
};

// Exchange buffers: U[c][m][g] = mode m of component c in warp c's own frame, P[v][g] = pressure at
// vertex v (the FP64 bits, after phase 1b the fixed-point value), biased exponents of the largest
// |u| and |p| that each warp saw.
struct OuterShared {
    long long U[3][27][kOuterCells];
    long long P[8][kOuterCells];
    int eu[3][kOuterCells], ep[3][kOuterCells];
};

__host__ __device__ __forceinline__ bool outer_bnd(int g, int M) { return g == 0 || g == M - 1; }

__host__ __device__ __forceinline__ void outer_atomic_add(double* p, double v) {
#ifdef __CUDA_ARCH__
    atomicAdd(p, v);
#else
    *p += v;
#endif
}

// ---- fixed point
constexpr int kFixBits = 54;      // |X| <= 2^54
constexpr int kFixMid = 12;       // bits dropped after the element matrix
constexpr int kFixMinExp = 64;    // below this largest exponent a zero does not fall out of fix_round by itself
constexpr int kFixLift = 128;     // such cells are read times 2^128; subnormal values read as 0
constexpr int kFixNone = -4096;   // exponent of a cell that reads as 0

__host__ __device__ __forceinline__ double bits_to_dbl(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double d;
    __builtin_memcpy(&d, &b, sizeof d);
    return d;
#endif
}
__host__ __device__ __forceinline__ long long mul_hi(long long a, long long b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (long long)(((__int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ unsigned long long mul_hi_u(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ int clz_u64(unsigned long long x) {   // x > 0
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}
__host__ __device__ __forceinline__ int exp_of(long long bits) { return int(bits >> 52) & 0x7FF; }

// X = round(v 2^(54 - E)) for the FP64 bits of v, |v| < 2^E with E = emax - 1022 (emax >= kFixMinExp,
// the largest biased exponent of the cell; cells below that: fix_lift). Zero, and what is below 2^-60 of the largest, gives 0.
__host__ __device__ __forceinline__ long long fix_round(long long bits, int emax) {
    const unsigned long long m = (unsigned long long)(bits & 0xFFFFFFFFFFFFFLL) << 2 | (1ull << 54);
    const int r = emax - exp_of(bits);
    const long long X = (long long)(((m >> (r < 60 ? r : 60)) + 1) >> 1);
    const long long s = bits >> 63;
    return (X ^ s) - s;
}

// x scale with x rounded to 53 bits (half up), |x| < 2^63: the significand is placed by integer
// instructions (from exponent scale.base), one FP64 multiplication.
struct FixScale {
    double s = 0.0;
    int base = 1085;
};
__host__ __device__ __forceinline__ double fix_out(long long x, const FixScale& scale) {
    const long long sign = x >> 63;
    const unsigned long long a = (unsigned long long)((x ^ sign) - sign);
    const int lz = a ? clz_u64(a) : 0;
    const unsigned long long v = a << lz;
    const long long m = (long long)((v >> 11) + ((v >> 10) & 1));
    const long long b = a ? m + ((long long)(scale.base - lz) << 52) : 0;   // m in [2^52, 2^53]: |x| = m 2^(11 - lz)
    return bits_to_dbl(b | (sign & (long long)(1ull << 63))) * scale.s;
}
// s 2^e, |e| < 3066; NaN where the cell holds one (or an infinity). A pressure against a large or small viscosity can
// take 2^e alone out of the FP64 range: three factors. For small values fix_out places |x| < 2^63 below 2, so that
// the factor is a normal number where the results can be.
__host__ __device__ __forceinline__ FixScale fix_scale(double s, int e, bool zero, bool bad) {
    FixScale r;
    if (bad) r.s = bits_to_dbl(0x7FF8000000000000LL);
    if (bad || zero) return r;
    if (e < -500) {
        r.base -= 62;
        e += 62;
    }
    int k = 0;
    if (e < -1022 || e > 1023) {
        k = e / 3;
        const double f = bits_to_dbl((long long)(k + 1023) << 52);
        s = s * f * f;
        k *= 2;
    }
    r.s = s * bits_to_dbl((long long)(e - k + 1023) << 52);
    return r;
}
// The FP64 bits of a value of a cell with largest exponent emax < kFixMinExp, times 2^128.
__host__ __device__ __forceinline__ long long fix_lift(long long bits) {
    return exp_of(bits) ? bits + ((long long)kFixLift << 52) : 0;
}
// B^T's factor (h^2 / 864) / s = km 2^(ek - 1084), km in [2^61, 2^62), to 2^-57. The result is multiplied by s, whose
// roundings would be the whole cell's if the factor did not take them back. In integers (Newton's iteration for 1/s
// from a single-precision start): the Stokes operator takes 23.6 us at 20^3 and 197 us at 64^3, 23.6 and 195 us with an
// FP64 division and its rounding; the division with its remainder in FP64 took 26.6 instead of 24.6 us at 20^3.
__host__ __device__ __forceinline__ long long fix_factor(double s, double h, int& ek) {
    const unsigned long long one = 1ull << 52;
    const long long sb = (long long)q2::dbl_bits(s), hb = (long long)q2::dbl_bits(h);
    const unsigned long long sm = (unsigned long long)(sb & (long long)(one - 1)) | (exp_of(sb) ? one : 0ull);
    const int lz = sm ? clz_u64(sm) : 0;                       // 11, more where s is subnormal
    const unsigned long long S = sm << lz;                     // s = S 2^(es - 1086)
    const int es = (exp_of(sb) ? exp_of(sb) : 1) + 11 - lz;
    unsigned long long X = (unsigned long long)(0x1p125f / float(S));   // 2^125 / S
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const long long err = (long long)((1ull << 61) - mul_hi_u(S, X));
        X += (unsigned long long)mul_hi((long long)X, err << 3);
    }
    const unsigned long long H = ((unsigned long long)(hb & (long long)(one - 1)) | one) << 11;
    const unsigned long long T = mul_hi_u(mul_hi_u(H, H), 0x97B425ED097B425Eull);   // 2^68 / 27
    const unsigned long long K = mul_hi_u(T, X);               // in [2^58, 2^62)
    const int sh = K ? clz_u64(K) - 2 : 0;
    ek = 2 * exp_of(hb) - es - sh - 8;
    return (long long)(K << sh);
}
// A 96-bit sum of products of modes with non-negative table entries below 2^12: high and low words apart.
struct FixSum {
    long long hi = 0;
    unsigned long long lo = 0;
    __host__ __device__ __forceinline__ void add(int c, long long u) {
        hi += (long long)c * int(u >> 32);
        lo += (unsigned long long)unsigned(c) * unsigned(u);
    }
    __host__ __device__ __forceinline__ long long shifted() const {
        return (hi << (32 - kFixMid)) + (long long)(lo >> kFixMid);
    }
};

// 97200 A in the modes, own component along local axis 0 (mode_diag and mode_cross as integers).
__host__ __device__ constexpr int fix_stiff(int a) { return a == 0 ? 0 : (a == 1 ? 3 : 4); }
__host__ __device__ constexpr int fix_mass(int a) { return a == 0 ? 5 : (a == 1 ? 15 : 4); }
__host__ __device__ constexpr int fix_diag(int i, int j, int k) {
    return 2 * fix_stiff(i) * fix_mass(j) * fix_mass(k) + fix_mass(i) * fix_stiff(j) * fix_mass(k) +
           fix_mass(i) * fix_mass(j) * fix_stiff(k);
}
__host__ __device__ constexpr int fix_cross(int a, int b, int o) { return 15 * (a + 1) * b * fix_mass(o); }

template <int AX>
__host__ __device__ __forceinline__ void fix_to_modes(long long* x) {
#pragma unroll
    for (int o2 = 0; o2 < 3; ++o2)
#pragma unroll
        for (int o1 = 0; o1 < 3; ++o1) {
            long long &a0 = x[q2::lin<AX>(0, o1, o2)], &a1 = x[q2::lin<AX>(1, o1, o2)], &a2 = x[q2::lin<AX>(2, o1, o2)];
            const long long s = a0 + a2, d = a2 - a0, m = a1;
            a0 = s + 4 * m;
            a1 = d;
            a2 = s - 2 * m;
        }
}
template <int AX>
__host__ __device__ __forceinline__ void fix_from_modes(long long* x) {
#pragma unroll
    for (int o2 = 0; o2 < 3; ++o2)
#pragma unroll
        for (int o1 = 0; o1 < 3; ++o1) {
            long long &w = x[q2::lin<AX>(0, o1, o2)], &d = x[q2::lin<AX>(1, o1, o2)], &e = x[q2::lin<AX>(2, o1, o2)];
            const long long t = w + e, a1 = 2 * (2 * w - e), dd = d;
            w = t - dd;
            d = a1;
            e = t + dd;
        }
}

// Every thread runs the same code: in its local frame the axes are rotated cyclically so that
// its own velocity component C lies along local axis 0 (local axes = global axes C, C+1, C+2
// mod 3). The operator is invariant under this relabelling (same 1D matrices and weights on every
// axis), so only the addressing differs between the three warps: gathers and scatters map local
// indices to global ones at run time, and warp C finds mode (i, j, k) of component C + 1 in that
// warp's frame at (j, k, i), of component C + 2 at (k, i, j). This keeps one copy of
// the unrolled code in the instruction cache.
struct OuterFrame {
    int C;            // velocity component of this thread
    size_t sn[3];     // global node strides of local axes 0, 1, 2
    int cl[3];        // cell coordinates along the local axes
    int ci, cj, ck;   // global cell coordinates
};

__host__ __device__ __forceinline__ OuterFrame outer_frame(const OuterArgs& a, int C, size_t cell) {
    OuterFrame f;
    f.C = C;
    f.ci = int(cell % a.n);
    f.cj = int((cell / a.n) % a.n);
    f.ck = int(cell / (size_t(a.n) * a.n));
    const size_t M = size_t(a.M);
#pragma unroll
    for (int d = 0; d < 3; ++d) {   // selects, not indexed arrays: those would live in local memory
        const int ax = (C + d) % 3;
        f.sn[d] = ax == 0 ? 1 : (ax == 1 ? M : M * M);
        f.cl[d] = ax == 0 ? f.ci : (ax == 1 ? f.cj : f.ck);
    }
    return f;
}

__host__ __device__ __forceinline__ size_t outer_vertex(const OuterArgs& a, const OuterFrame& f, int gv) {
    const int P = a.n + 1;
    return size_t(f.ci + (gv & 1)) + size_t(P) * (f.cj + ((gv >> 1) & 1) + size_t(P) * (f.ck + (gv >> 2)));
}

// Phase 1: gather the own component (raw FP64 bits, kept in T for phase 1b) and every third
// pressure vertex, and the largest exponents. V is any 8-byte type; U is the caller's scratch and not used.
template <bool DO_A, bool DO_B, bool DO_BT = true, typename V>
__host__ __device__ __forceinline__ void outer_phase1(const OuterArgs& a, int C, int blk, int g, OuterShared& sh,
                                                      V (&U)[27], V (&T)[27]) {
    static_assert(sizeof(V) == 8, "an 8-byte slot per value");
    (void)U;
    const size_t cells = size_t(a.n) * a.n * a.n;
    const size_t cell = size_t(blk) * kOuterCells + g;
    const bool valid = cell < cells;
    const OuterFrame f = outer_frame(a, C, valid ? cell : 0);
    if (DO_A || DO_B) {
        const double* src = a.src_u + size_t(C) * a.nodes +
                            (size_t(2 * f.ci) + size_t(a.M) * (size_t(2 * f.cj) + size_t(a.M) * size_t(2 * f.ck)));
        int e = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int b = 0; b < 3; ++b)
#pragma unroll
                for (int aa = 0; aa < 3; ++aa) {
                    const bool bnd = !valid || outer_bnd(2 * f.cl[0] + aa, a.M) || outer_bnd(2 * f.cl[1] + b, a.M) ||
                                     outer_bnd(2 * f.cl[2] + c, a.M);
                    const double v = bnd ? 0.0 : src[aa * f.sn[0] + b * f.sn[1] + c * f.sn[2]];
                    const int ev = exp_of((long long)q2::dbl_bits(v));
                    e = ev > e ? ev : e;
                    memcpy(&T[aa + 3 * b + 9 * c], &v, 8);
                }
        sh.eu[C][g] = e;
    }
    if (DO_BT) {
        int e = 0;
        for (int v = C; v < 8; v += 3) {
            const double p = valid ? a.src_p[outer_vertex(a, f, v)] : 0.0;
            const long long b = (long long)q2::dbl_bits(p);
            e = exp_of(b) > e ? exp_of(b) : e;
            sh.P[v][g] = b;
        }
        sh.ep[C][g] = e;
    }
}

__host__ __device__ __forceinline__ int max3(const int (&e)[3][kOuterCells], int g) {
    const int m = e[0][g] > e[1][g] ? e[0][g] : e[1][g];
    return m > e[2][g] ? m : e[2][g];
}

// This thread's component (raw FP64 bits T) in fixed point against the cell's largest magnitude, and its
// modes; every third pressure value (sh.P) in fixed point. After the barrier behind sh.eu and sh.ep.
template <bool DO_U, bool DO_P, typename V>
__host__ __device__ __forceinline__ void outer_modes(int C, int g, OuterShared& sh, V (&T)[27]) {
    if (DO_U) {
        int e = max3(sh.eu, g);
        if (e < kFixMinExp) {
            e += kFixLift;
#pragma unroll
            for (int m = 0; m < 27; ++m) {
                long long b;
                memcpy(&b, &T[m], 8);
                b = fix_lift(b);
                memcpy(&T[m], &b, 8);
            }
        }
        long long X[27];
#pragma unroll
        for (int m = 0; m < 27; ++m) {
            long long b;
            memcpy(&b, &T[m], 8);
            X[m] = fix_round(b, e);
        }
        fix_to_modes<0>(X);
        fix_to_modes<1>(X);
        fix_to_modes<2>(X);
#pragma unroll
        for (int m = 0; m < 27; ++m) sh.U[C][m][g] = X[m];
    }
    if (DO_P) {
        const int e = max3(sh.ep, g);
        for (int v = C; v < 8; v += 3)
            sh.P[v][g] = e < kFixMinExp ? fix_round(fix_lift(sh.P[v][g]), e + kFixLift) : fix_round(sh.P[v][g], e);
    }
}

// B u of a cell of side h at its vertices (warp C's frame: bit d of the index along global axis C + d), as
// b scale. After the barrier behind outer_modes.
__host__ __device__ __forceinline__ FixScale outer_pressure(int C, int g, const OuterShared& sh, double h, long long (&b)[8]) {
    const int D1 = (C + 1) % 3, D2 = (C + 2) % 3, eu = max3(sh.eu, g);
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const int i = v & 1, j = (v >> 1) & 1, k = v >> 2;
        b[v] = ((3 - i) * sh.U[C][(i + 1) + 3 * j + 9 * k][g] >> 2) + ((3 - j) * sh.U[D1][(j + 1) + 3 * k + 9 * i][g] >> 2) +
               ((3 - k) * sh.U[D2][(k + 1) + 3 * i + 9 * j][g] >> 2);
    }
    q2::from_pressure_modes(b);
    return fix_scale(-h * h / 864.0, eu - 1022 - kFixBits + 2, eu == 0, eu == 0x7FF);
}

// Component C of A u + B^T p of a cell of side h and viscosity mu, in warp C's frame, as Y scale.
template <bool DO_A, bool DO_BT>
__host__ __device__ __forceinline__ FixScale outer_velocity(int C, int g, const OuterShared& sh, double mu, double h,
                                                            long long (&Y)[27]) {
    const int D1 = (C + 1) % 3, D2 = (C + 2) % 3;
    const int eu = DO_A ? max3(sh.eu, g) : 0;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int m = i + 3 * j + 9 * k;
                FixSum y;
                if (DO_A) {
                    if (m != 0) y.add(fix_diag(i, j, k), sh.U[C][m][g]);
                    if (i < 2 && j > 0) y.add(fix_cross(i, j, k), sh.U[D1][(j - 1) + 3 * k + 9 * (i + 1)][g]);
                    if (i < 2 && k > 0) y.add(fix_cross(i, k, j), sh.U[D2][(k - 1) + 3 * (i + 1) + 9 * j][g]);
                }
                Y[m] = y.shifted();
            }
    const double s = mu * h * (1.0 / 97200.0);
    const int eu0 = DO_A && eu > 0 ? eu : kFixNone;
    int E = eu0;
    bool bad = DO_A && eu == 0x7FF;
    if (DO_BT) {
        // p' = 112.5 h/mu p: the vertex modes times the factor's significand, |R| <= 2^60; |p'| < 2^(epk - 1022)
        // may exceed |u| by 2^10 before its share of the result is the larger one
        const int ep = max3(sh.ep, g);
        if (ep > 0) {
            int ek;
            const long long km = fix_factor(s, h, ek);
            const int epk = ep + ek - 1022;
            E = E > epk - 10 ? E : epk - 10;
            long long P[8];
#pragma unroll
            for (int v = 0; v < 8; ++v)
                P[v] = sh.P[((v & 1) << C) + (((v >> 1) & 1) << D1) + ((v >> 2) << D2)][g];
            q2::to_pressure_modes(P);
            const int sp = E - epk + 15 < 63 ? E - epk + 15 : 63;
            const int sa = DO_A ? (E - eu0 < 63 ? E - eu0 : 63) : 0;
            if (sa > 0) {
#pragma unroll
                for (int m = 0; m < 27; ++m) Y[m] >>= sa;
            }
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const int i = v & 1, j = (v >> 1) & 1, k = v >> 2;
                Y[(i + 1) + 3 * j + 9 * k] -= (3 - i) * (mul_hi(P[v] * 32, km) >> sp);
            }
            bad = bad || ep == 0x7FF;
        }
    }
    fix_from_modes<2>(Y);
    fix_from_modes<1>(Y);
    fix_from_modes<0>(Y);
    return fix_scale(s, E - 1022 - kFixBits + kFixMid, E == kFixNone, bad);
}

// Phase 1b (after a barrier): fixed point and modes.
template <bool DO_A, bool DO_B = true, bool DO_BT = true, typename V>
__host__ __device__ __forceinline__ void outer_phase1b(const OuterArgs&, int C, int, int g, OuterShared& sh,
                                                       V (&T)[27]) {
    outer_modes<DO_A || DO_B, DO_BT>(C, g, sh, T);
}

// Phase 2 (after a barrier): the element matrix in the modes, the transposed transform and the
// scatter into the velocity output; B u at this warp's vertices.
template <bool DO_A, bool DO_BT, bool DO_B = true, typename V>
__host__ __device__ __forceinline__ void outer_phase2(const OuterArgs& a, int C, int blk, int g, const OuterShared& sh,
                                                      V (&W)[27]) {
    (void)W;
    const size_t cells = size_t(a.n) * a.n * a.n;
    const size_t cell = size_t(blk) * kOuterCells + g;
    if (cell >= cells) return;
    const OuterFrame f = outer_frame(a, C, cell);
    if (DO_B) {
        long long b[8];
        const FixScale s = outer_pressure(C, g, sh, a.h, b);
        // the vertex one step along the own axis and its opposite; the two that no rotation moves
        // go to warps 0 and 1
        outer_atomic_add(a.dst_p + outer_vertex(a, f, 1 << C), fix_out(b[1], s));
        outer_atomic_add(a.dst_p + outer_vertex(a, f, 7 - (1 << C)), fix_out(b[6], s));
        if (C < 2) outer_atomic_add(a.dst_p + outer_vertex(a, f, C == 0 ? 0 : 7), fix_out(C == 0 ? b[0] : b[7], s));
    }
    if (!(DO_A || DO_BT)) return;
    long long Y[27];
    const FixScale s = outer_velocity<DO_A, DO_BT>(C, g, sh, a.mu[cell], a.h, Y);
    double* dst = a.dst_u + size_t(C) * a.nodes +
                  (size_t(2 * f.ci) + size_t(a.M) * (size_t(2 * f.cj) + size_t(a.M) * size_t(2 * f.ck)));
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int aa = 0; aa < 3; ++aa) {
                const int g0 = 2 * f.cl[0] + aa, g1 = 2 * f.cl[1] + b, g2 = 2 * f.cl[2] + c;
                if (outer_bnd(g0, a.M) || outer_bnd(g1, a.M) || outer_bnd(g2, a.M)) continue;
                outer_atomic_add(dst + aa * f.sn[0] + b * f.sn[1] + c * f.sn[2], fix_out(Y[aa + 3 * b + 9 * c], s));
            }
}

}  // namespace stk
