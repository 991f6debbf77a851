// Host walk through the sweeps of the double-float Gram-Schmidt passes (csrc/gs.cuh, the loop of k_gs_df).
// Test support only: tests/test_gs_host.py.
#include <cstddef>
#include <vector>

#include "df64.cuh"
#include "gs.cuh"

// For rows of n entries, `blocks` CTAs and tpe threads to a pair: the first pair whose rows threads of more than one
// group of tpe, or of more than one sweep, read, np if a pair is left out, -1 if each is read by its own group only.
extern "C" long long gs_shared_pair(size_t n, unsigned blocks, int tpe) {
    using namespace stk;
    const size_t np = (n + 1) / 2, stride = size_t(blocks) * unsigned(kGsThreads / tpe);
    std::vector<long long> owner(np, -1);
    for (unsigned b = 0; b < blocks; ++b)
        for (int t = 0; t < kGsThreads; ++t) {
            const size_t warp_first = gs_pair(0, b, t / 32 * 32, tpe);
            for (size_t base = 0; warp_first + base < np; base += stride) {
                const size_t p = gs_pair(base, b, t, tpe);
                if (!gs_reads(p, np)) continue;
                if (p >= np) return (long long)np;
                const long long who = (long long)((base / stride * blocks + b) * kGsThreads + t / tpe);
                if (owner[p] >= 0 && owner[p] != who) return (long long)p;
                owner[p] = who;
            }
        }
    for (size_t p = 0; p < np; ++p)
        if (owner[p] < 0) return (long long)np;
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
