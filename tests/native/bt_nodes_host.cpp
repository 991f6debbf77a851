// Host run of B^T p as k_bt forms it (csrc/pressure.cuh bt_nodes): the 8 lower and odd nodes of every
// cell, in FP64 and in double-float pairs. Test support only: tests/test_bt_nodes.py.
#include <algorithm>
#include <cstddef>

#include "pressure.cuh"

template <int C, typename T, typename In, typename Out>
static void component(int n, double h, const T (&v)[3][3][3], int e, int f, int g, double* out, In in, Out to) {
    const int M = 2 * n + 1;
    T b[8];
    stk::bt_nodes<C>(v, b);
    for (int q = 0; q < 8; ++q) {
        const int i = q & 1, j = (q >> 1) & 1, k = q >> 2;
        if ((i == 0 && e == 0) || (j == 0 && f == 0) || (k == 0 && g == 0)) continue;
        out[size_t(C) * M * M * M + size_t(2 * e + i) + size_t(M) * (2 * f + j + size_t(M) * (2 * g + k))] =
            to(b[q] * in(-h * h * stk::bt_factor<C>(i, j, k)));
    }
}

template <typename T, typename In, typename Out>
static void apply(int n, const double* p, double* out, In in, Out to) {
    const int P = n + 1, M = 2 * n + 1;
    const double h = 1.0 / n;
    for (size_t i = 0; i < 3 * size_t(M) * M * M; ++i) out[i] = 0.0;
    for (int g = 0; g < n; ++g)
        for (int f = 0; f < n; ++f)
            for (int e = 0; e < n; ++e) {
                T v[3][3][3];
                for (int k = 0; k < 3; ++k)
                    for (int j = 0; j < 3; ++j)
                        for (int i = 0; i < 3; ++i)
                            v[k][j][i] = in(p[size_t(std::max(e - 1 + i, 0)) +
                                              size_t(P) * (std::max(f - 1 + j, 0) + size_t(P) * std::max(g - 1 + k, 0))]);
                component<0>(n, h, v, e, f, g, out, in, to);
                component<1>(n, h, v, e, f, g, out, in, to);
                component<2>(n, h, v, e, f, g, out, in, to);
            }
}

extern "C" void bt_nodes_f64(int n, const double* p, double* out) {
    apply<double>(n, p, out, [](double x) { return x; }, [](double x) { return x; });
}
extern "C" void bt_nodes_df64(int n, const double* p, double* out) {
    apply<q2::df64>(n, p, out, [](double x) { return q2::split_double(x); }, [](const q2::df64& x) { return x.to_double(); });
}
