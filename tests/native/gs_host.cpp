// Host walk through the sweeps of the double-float Gram-Schmidt passes (csrc/gs.cuh, the loop of k_gs_df).
// Test support only: tests/test_gs_host.py.
#include <cstddef>
#include <vector>

#include "df64.cuh"
#include "gs.cuh"

// For k rows of n entries, `blocks` CTAs, tpe threads to a pair and rb rows to a thread: the first pair of row k - 1 that
// threads of more than one group of tpe, or in more than one sweep, read; np if some pair of some row is left
// out or something past the rows or pairs is read; -1 if neither.
extern "C" long long gs_shared_pair(size_t n, unsigned blocks, int tpe, int rb, int k) {
    using namespace stk;
    const size_t np = (n + 1) / 2, stride = size_t(blocks) * unsigned(kGsThreads / tpe);
    std::vector<long long> owner(np, -1);         // of row k - 1's pairs
    std::vector<char> seen(np * size_t(k), 0);   // pairs of all rows
    for (unsigned b = 0; b < blocks; ++b)
        for (int t = 0; t < kGsThreads; ++t) {
            const size_t warp_first = gs_pair(0, b, t / 32 * 32, tpe);
            for (size_t base = 0; warp_first + base < np; base += stride) {
                const size_t p = gs_pair(base, b, t, tpe);
                const size_t rp = gs_read_pair(p, np);
                const int r0 = t % tpe * rb, rows = gs_read_rows(p >= np, k, r0, rb);
                if (rp >= np || r0 + rows > k) return (long long)np;
                for (int r = 0; r < rows; ++r) seen[size_t(r0 + r) * np + rp] = 1;
                if (r0 + rows < k || rows == 0) continue;
                const long long who = (long long)((base / stride * blocks + b) * kGsThreads + t / tpe);
                if (owner[rp] >= 0 && owner[rp] != who) return (long long)rp;
                owner[rp] = who;
            }
        }
    for (char s : seen)
        if (!s) return (long long)np;
    return -1;
}

extern "C" double gs_small_limit() { return stk::kSmallC; }

// sum_i c[i] v[i] of one entry in the single-precision form of k_gs_df: lane g has rows g rb .. g rb + rb - 1, the
// lanes' sums are added as its shuffles add them.
extern "C" double gs_small_sum(int tpe, int rb, const double* c, const double* v) {
    float lane[4] = {};
    for (int g = 0; g < tpe; ++g)
        for (int r = 0; r < rb; ++r)
            lane[g] = stk::gs_small(float(c[g * rb + r]), q2::split_double(v[g * rb + r]).hi, lane[g]);
    for (int o = 1; o < tpe; o <<= 1) {
        float next[4];
        for (int g = 0; g < tpe; ++g) next[g] = lane[g] + lane[g ^ o];
        for (int g = 0; g < tpe; ++g) lane[g] = next[g];
    }
    return double(lane[0]);
}
