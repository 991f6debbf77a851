// march.cu -- the FP32 level operator (Section 2.1, definition of A) with its epilogue in one launch,
// without atomic adds: A x, b - A x, or the Jacobi-Chebyshev step of Section 2.2.1.
//
// A block owns a tile of 16 x 6 cells in x and y and marches over OZ cell layers, one thread per
// cell column. It also computes the column of cells before the tile along x and along y and the layer
// below its first, whose results complete the nodes that it owns: the nodes with local index 0 or 1
// in an owned cell. Per layer a thread
//   - reads the two new node planes of its cell (the lower one is the upper one of the layer before,
//     kept in modes along x and y) and forms the cell product in the modes of q2_basis.cuh;
//   - adds the upper plane of the layer before to its lower plane (again in modes along x and y:
//     the transposed transforms of a plane run once, not for both cells that share it);
//   - exchanges the nodes on its upper x and y sides with the neighbouring threads through shared
//     memory and runs the epilogue on its 24 nodes.
// The operand's rows come two layers ahead, the epilogue's operands one phase ahead, as 16-byte
// asynchronous copies into shared memory (through registers each layer waited for its loads twice;
// one bulk copy per row serialises over a warp's lanes, ~9 instructions each). Rows of a vector start
// at any 4-byte offset (M is odd): a copy starts at the 16-byte boundary below and the row is read at
// the remainder. The parity of a cell's row is known at compile time, so two of its three nodes are
// one 8-byte access.
#include "brick.cuh"
#include "prof.cuh"

#include <cstdint>

#define LAUNCH(cls, s, ...)              \
    do {                                \
        prof_begin((cls), (s));         \
        __VA_ARGS__;                    \
        prof_end((cls), (s));           \
        prof_count(1);                  \
    } while (0)

namespace stk {

namespace {

constexpr int kTileX = 16, kTileY = 6;                       // owned cells
constexpr int kColsX = kTileX + 1, kColsY = kTileY + 1;      // computed cells
constexpr int kMarchThreads = 128;                           // 119 columns
constexpr int kRowX = 40;                                    // 35 nodes, up to 3 before them; entries per copied row
constexpr int kRowsX = 2 * kColsY + 1;                       // node rows of a plane
constexpr int kRowE = 36;                                    // 32 owned nodes, up to 3 before them
constexpr int kXRows = 3 * 2 * kRowsX;                       // rows per layer: components, two planes
constexpr int kERows = 3 * 2 * 2 * kTileY;                   // owned rows per layer and operand
constexpr int kPassX = kMarchThreads / (kRowX / 4);          // rows of a plane that the block copies at a time
static_assert(2 * kTileY * (kRowE / 4) <= kMarchThreads, "one 16-byte copy per thread and plane of an operand");

struct MarchArgs {
    int n, M;
    int oz;                // cell layers owned by a block
    size_t nodes;
    float h;
    const float* mu;
    const float* src;      // operand x
    float* dst;            // EPI_PLAIN: A x; EPI_RESID: b - A x; EPI_CHEB: the new x (not src)
    const float* b;
    const float* dinv;
    const float* d;        // EPI_CHEB: the direction
    float* d_new;          // EPI_CHEB: the new direction (not d: the copies of a row reach into the next tile's)
    float c1, c2;
};

template <int EPI>
struct MarchShared {
    static constexpr int NE = EPI == EPI_CHEB ? 4 : (EPI == EPI_RESID ? 1 : 0);   // b, dinv, d, x
    float X[2][kXRows][kRowX];
    float E[NE > 0 ? NE : 1][NE > 0 ? kERows : 1][kRowE];
    float ex[30][kMarchThreads];
};

__device__ __forceinline__ void copy16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(unsigned(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The three nodes of an x-row, parity = offset of the first from an 8-byte boundary in entries.
template <int PARITY>
__device__ __forceinline__ void load_row3(const float* p, float (&v)[3]) {
    if (PARITY == 0) {
        const float2 a = *reinterpret_cast<const float2*>(p);
        v[0] = a.x;
        v[1] = a.y;
        v[2] = p[2];
    } else {
        v[0] = p[0];
        const float2 a = *reinterpret_cast<const float2*>(p + 1);
        v[1] = a.x;
        v[2] = a.y;
    }
}
template <int PARITY>
__device__ __forceinline__ float2 load_pair(const float* p) {
    return PARITY == 0 ? *reinterpret_cast<const float2*>(p) : make_float2(p[0], p[1]);
}
template <int PARITY>
__device__ __forceinline__ void store_pair(float* p, float2 v) {
    if (PARITY == 0) {
        *reinterpret_cast<float2*>(p) = v;
    } else {
        p[0] = v.x;
        p[1] = v.y;
    }
}

// Which nodes of a thread's cell read as 0: bit 0 / 2 the first / last along x, bits 3, 5 along y; 64: all.
constexpr int kZx0 = 1, kZx2 = 4, kZy0 = 8, kZy2 = 32, kZAll = 64;

// The rows r[j] of one plane, masked, to modes along x and y.
__device__ __forceinline__ void plane_modes(float (&r)[3][3], int zero, bool live, float* x) {
    if (zero != 0 || !live) {
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int m = kZAll | (i == 0 ? kZx0 : i == 2 ? kZx2 : 0) | (j == 0 ? kZy0 : j == 2 ? kZy2 : 0);
                if (!live || (zero & m)) r[j][i] = 0.0f;
            }
    }
    float q[9];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float s = r[j][0] + r[j][2];
        q[3 * j] = s + 4.0f * r[j][1];
        q[3 * j + 1] = r[j][2] - r[j][0];
        q[3 * j + 2] = s - 2.0f * r[j][1];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float s = q[i] + q[6 + i];
        x[i] = s + 4.0f * q[3 + i];
        x[3 + i] = q[6 + i] - q[i];
        x[6 + i] = s - 2.0f * q[3 + i];
    }
}
// Plane P (0: the odd one, 1: the even one above it) of component C from the copied rows at x (the
// thread's first node, without the remainder rem[(C + j) mod 4] of row j).
template <int C, int P>
__device__ __forceinline__ void tile_plane(const float* x, const int (&rem)[4], int zero, bool live, float* out) {
    float r[3][3];
    const float* p = x + (2 * C + P) * (kRowsX * kRowX);
    load_row3<(C + P + 1) & 1>(p + rem[C & 3], r[0]);
    load_row3<(C + P) & 1>(p + rem[(C + 1) & 3] + kRowX, r[1]);
    load_row3<(C + P + 1) & 1>(p + rem[(C + 2) & 3] + 2 * kRowX, r[2]);
    plane_modes(r, zero, live, out);
}
// The even plane below a block's first layer, straight from memory.
template <int C>
__device__ __forceinline__ void first_plane(const float* p, int M, int zero, bool live, float* out) {
    float r[3][3] = {{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}};
    if (live && !(zero & kZAll)) {
        load_row3<C & 1>(p, r[0]);
        load_row3<(C + 1) & 1>(p + M, r[1]);
        load_row3<C & 1>(p + 2 * M, r[2]);
    }
    plane_modes(r, zero, live, out);
}
// Transposed: modes along x and y of one plane to its nodes.
__device__ __forceinline__ void plane_nodes(float* x) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float w = x[i], d = x[3 + i], e = x[6 + i], t = w + 0.5f * e;
        x[i] = t - d;
        x[3 + i] = 4.0f * w - e;
        x[6 + i] = t + d;
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float w = x[3 * j], d = x[3 * j + 1], e = x[3 * j + 2], t = w + 0.5f * e;
        x[3 * j] = t - d;
        x[3 * j + 1] = 4.0f * w - e;
        x[3 * j + 2] = t + d;
    }
}

// Row component C: element matrix, z transform, the share of the layer below; the lower two planes
// become nodal values: the own four nodes of each into S, the five on the upper sides into ex.
template <int C>
__device__ __forceinline__ void march_row(const float* U, const float* U1, const float* U2, float s, float* carry,
                                          bool out, float (&S)[3][2][4], float (*ex)[kMarchThreads], int t) {
    float w[27];
    q2::modes_A<C>(U, U1, U2, w);
#pragma unroll
    for (int m = 0; m < 27; ++m) w[m] *= s;
    q2::from_modes<2>(w);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        w[q] += carry[q];
        carry[q] = w[18 + q];
    }
    if (!out) return;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        float* x = w + 9 * p;
        plane_nodes(x);
        S[C][p][0] = x[0];
        S[C][p][1] = x[1];
        S[C][p][2] = x[3];
        S[C][p][3] = x[4];
        float(*e)[kMarchThreads] = ex + 10 * C + 5 * p;
        e[0][t] = x[2];
        e[1][t] = x[5];
        e[2][t] = x[6];
        e[3][t] = x[7];
        e[4][t] = x[8];
    }
}

// Two nodes of an owned row: ax the complete product, e their place in the copied row of operand 0
// (the same in the other operands' rows), i their place in the vectors.
template <int EPI, int PARITY>
__device__ __forceinline__ void march_epilogue(const MarchArgs& a, const float* e, size_t i, float2 ax) {
    constexpr int kNext = kERows * kRowE;   // the next operand's row
    if constexpr (EPI == EPI_PLAIN) {
        store_pair<PARITY>(a.dst + i, ax);
    } else {
        const float2 b = load_pair<PARITY>(e);
        if constexpr (EPI == EPI_RESID) {
            store_pair<PARITY>(a.dst + i, make_float2(b.x - ax.x, b.y - ax.y));
        } else {
            const float2 di = load_pair<PARITY>(e + kNext), d = load_pair<PARITY>(e + 2 * kNext),
                         x = load_pair<PARITY>(e + 3 * kNext);
            const bool old = a.c1 != 0.0f;   // a first step has no direction before it: d holds anything, NaN too
            const float2 dn = make_float2((old ? a.c1 * d.x : 0.0f) + a.c2 * (di.x * (b.x - ax.x)),
                                          (old ? a.c1 * d.y : 0.0f) + a.c2 * (di.y * (b.y - ax.y)));
            store_pair<PARITY>(a.d_new + i, dn);
            store_pair<PARITY>(a.dst + i, make_float2(x.x + dn.x, x.y + dn.y));
        }
    }
}

// Own nodes of component C in plane P (0: even, 1: odd): the neighbours' shares, then the epilogue on
// two rows of two; 0 on constrained nodes (first column x0, first row y0). e: the thread's first
// owned node in the copied rows, without the remainder.
template <int EPI, int C, int P>
__device__ __forceinline__ void march_own(const MarchArgs& a, const float* e, const float (*ex)[kMarchThreads],
                                          const float (&S)[3][2][4], int t, const int (&rem)[4], size_t i, bool x0, bool y0) {
    const float(*n)[kMarchThreads] = ex + 10 * C + 5 * P;
    float2 r0 = make_float2(S[C][P][0] + n[0][t - 1] + n[2][t - kColsX] + n[4][t - kColsX - 1],
                            S[C][P][1] + n[3][t - kColsX]);
    float2 r1 = make_float2(S[C][P][2] + n[1][t - 1], S[C][P][3]);
    if (x0 || y0) r0.x = 0.0f;
    if (y0) r0.y = 0.0f;
    if (x0) r1.x = 0.0f;
    const float* row = e + (2 * C + P) * (2 * kTileY * kRowE);
    march_epilogue<EPI, (C + P) & 1>(a, row + rem[C & 3], i, r0);
    march_epilogue<EPI, (C + P + 1) & 1>(a, row + rem[(C + 1) & 3] + kRowE, i + a.M, r1);
}

template <int EPI>
__global__ void __launch_bounds__(kMarchThreads, 2) k_march(MarchArgs a) {
    extern __shared__ __align__(128) unsigned char march_smem[];
    MarchShared<EPI>& sh = *reinterpret_cast<MarchShared<EPI>*>(march_smem);
    constexpr int NE = MarchShared<EPI>::NE;
    const int t = threadIdx.x, n = a.n, M = a.M, Mq = M & 3;
    const int tx = t % kColsX, ty = t / kColsX;
    const int ci = int(blockIdx.x) * kTileX + tx - 1, cj = int(blockIdx.y) * kTileY + ty - 1;
    const bool valid = ci >= 0 && cj >= 0 && ci < n && cj < n && ty < kColsY;
    const bool own = valid && tx > 0 && ty > 0;
    const int z0 = int(blockIdx.z) * a.oz, z1 = min(n, z0 + a.oz), kb = z0 > 0 ? z0 - 1 : 0;
    const int zero = !valid ? kZAll
                            : (ci == 0 ? kZx0 : 0) | (ci == n - 1 ? kZx2 : 0) | (cj == 0 ? kZy0 : 0) | (cj == n - 1 ? kZy2 : 0);
    const size_t MM = size_t(M) * M;
    // first node column and row of the computed cells; the owned ones start two further
    const int ix = 2 * (int(blockIdx.x) * kTileX - 1), jx = 2 * (int(blockIdx.y) * kTileY - 1);
    // Copies of the operand's planes 2 ck + 1 and 2 ck + 2 (rows of them that are not constrained) into
    // buffer buf: thread t takes 16 bytes t % 10 of row t / 10 and of the row kPassX further.
    const int xj = t / (kRowX / 4), xc = 4 * (t % (kRowX / 4));
    auto issue_x = [&](int ck, int buf) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const float* plane = a.src + (size_t(c) * a.nodes + MM * size_t(2 * ck + 1 + p));
                if (p == 1 && ck == n - 1) continue;
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const int r = xj + m * kPassX, j = jx + r;
                    if (r >= (m == 0 ? kPassX : kRowsX) || j < 1 || j >= M - 1) continue;
                    const int rem = (ix + (c + j) * Mq + 2 * ck + 1 + p) & 3;
                    copy16(&sh.X[buf][(2 * c + p) * kRowsX + r][xc], plane + (ix + M * j - rem + xc));
                }
            }
    };
    // Copies of the epilogue's operands on the owned rows of planes 2 ck and 2 ck + 1 (the plane 0 is
    // constrained): 16 bytes t % 9 of row t / 9.
    const int ej = t / (kRowE / 4), ec = 4 * (t % (kRowE / 4));
    const bool e_row = ej < 2 * kTileY && jx + 2 + ej < M - 1;
    auto issue_e = [&](int ck) {
        if (!e_row) return;
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (p == 0 && ck == 0) continue;
                const int j = jx + 2 + ej, rem = (ix + 2 + (c + j) * Mq + 2 * ck + p) & 3;
                const size_t at = size_t(c) * a.nodes + MM * size_t(2 * ck + p) + size_t(ix + 2 + M * j - rem + ec);
#pragma unroll
                for (int k = 0; k < NE; ++k)
                    copy16(&sh.E[k][(2 * c + p) * (2 * kTileY) + ej][ec], (k == 0 ? a.b : (k == 1 ? a.dinv : (k == 2 ? a.d : a.src))) + at);
            }
    };
    issue_x(kb, 0);
    copy_commit();
    if (kb + 1 < z1) issue_x(kb + 1, 1);
    if constexpr (NE > 0) issue_e(z0);
    copy_commit();
    size_t base = valid ? size_t(2 * ci) + size_t(M) * size_t(2 * cj) + MM * size_t(2 * kb) : 0;
    const float* mu = a.mu + (valid ? size_t(ci) + size_t(n) * (size_t(cj) + size_t(n) * kb) : 0);
    float low[3][9], carry[3][9];
    {
        const float* s0 = a.src + base;
        const bool live = kb > 0;
        first_plane<0>(s0, M, zero, live, low[0]);
        first_plane<1>(s0 + a.nodes, M, zero, live, low[1]);
        first_plane<2>(s0 + 2 * a.nodes, M, zero, live, low[2]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int q = 0; q < 9; ++q) carry[c][q] = 0.0f;
    // Remainders mod 4 of this thread's rows (vectors are 16-byte aligned; M^2 = 1 and M^3 = M mod 4): row j
    // of component c lies (c + j) M further, the odd plane 1, a layer 2. ev, od: the owned nodes in the
    // even and odd plane of the layer; the operand's tile starts two nodes before them.
    int ev[4], od[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        ev[k] = (ix + 2 + (jx + 2 * ty + k) * Mq + 2 * kb) & 3;
        od[k] = (ev[k] + 1) & 3;
    }
    copy_wait<1>();
    __syncthreads();
    const float* const tile = &sh.X[0][0][0] + min(ty, kColsY - 1) * 2 * kRowX + 2 * tx;
    const float* const oper = &sh.E[0][0][0] + (2 * (ty - 1)) * kRowE + 2 * (tx - 1);   // used by owners only
    float mu_next = valid ? *mu : 0.0f;   // a layer ahead: its latency is not waited for
#pragma unroll 1
    for (int ck = kb; ck < z1; ++ck) {
        const int it = ck - kb;
        float U[3][27];
        const float s = mu_next * a.h;
        mu += size_t(n) * n;
        if (valid && ck + 1 < z1) mu_next = *mu;
        {
            const float* x = tile + (it & 1) * (kXRows * kRowX);
            const bool top = ck < n - 1;
            const int od2[4] = {od[0] ^ 2, od[1] ^ 2, od[2] ^ 2, od[3] ^ 2};
            tile_plane<0, 0>(x, od2, zero, true, U[0] + 9);
            tile_plane<1, 0>(x, od2, zero, true, U[1] + 9);
            tile_plane<2, 0>(x, od2, zero, true, U[2] + 9);
            tile_plane<0, 1>(x, ev, zero, top, U[0] + 18);   // the next layer's even plane: twice two further
            tile_plane<1, 1>(x, ev, zero, top, U[1] + 18);
            tile_plane<2, 1>(x, ev, zero, top, U[2] + 18);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                U[c][q] = low[c][q];
                low[c][q] = U[c][18 + q];
            }
            q2::to_modes<2>(U[c]);
        }
        const bool out = ck >= z0;   // the same for the whole block
        float S[3][2][4];
        march_row<0>(U[0], U[1], U[2], s, carry[0], out, S, sh.ex, t);
        march_row<1>(U[1], U[2], U[0], s, carry[1], out, S, sh.ex, t);
        march_row<2>(U[2], U[0], U[1], s, carry[2], out, S, sh.ex, t);
        copy_wait<0>();    // the operands of this layer, the rows of the next one
        __syncthreads();   // ... and ex are complete, this layer's rows are read
        if (ck + 2 < z1) issue_x(ck + 2, it & 1);
        copy_commit();
        if (out) {
            if (own) {
                const bool x0 = ci == 0, y0 = cj == 0;
                if (ck > 0) {
                    march_own<EPI, 0, 0>(a, oper, sh.ex, S, t, ev, base, x0, y0);
                    march_own<EPI, 1, 0>(a, oper, sh.ex, S, t, ev, base + a.nodes, x0, y0);
                    march_own<EPI, 2, 0>(a, oper, sh.ex, S, t, ev, base + 2 * a.nodes, x0, y0);
                }
                march_own<EPI, 0, 1>(a, oper, sh.ex, S, t, od, base + MM, x0, y0);
                march_own<EPI, 1, 1>(a, oper, sh.ex, S, t, od, base + MM + a.nodes, x0, y0);
                march_own<EPI, 2, 1>(a, oper, sh.ex, S, t, od, base + MM + 2 * a.nodes, x0, y0);
            }
            if (ck + 1 < z1) {
                __syncthreads();   // ex and the operand rows are read
                if constexpr (NE > 0) issue_e(ck + 1);
                copy_commit();
            }
        }
        base += 2 * MM;
#pragma unroll
        for (int k = 0; k < 4; ++k) ev[k] ^= 2, od[k] ^= 2;
    }
}

template <int EPI>
cudaError_t march_config() {
    return cudaFuncSetAttribute(k_march<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(MarchShared<EPI>)));
}

}  // namespace

// Layers per block: the least layers (one more for the halo) times waves of two blocks per SM.
static int march_layers(int n) {
    const int tiles = ((n + kTileX - 1) / kTileX) * ((n + kTileY - 1) / kTileY);
    int best = 1 << 30, oz = n;
    for (int z = 1; z <= n; ++z) {
        const int blocks = tiles * ((n + z - 1) / z), layers = (blocks + 303) / 304 * (z + (z < n ? 1 : 0));
        if (layers < best) best = layers, oz = z;
    }
    return oz;
}

cudaError_t march_configure() {
    cudaError_t e;
    if ((e = march_config<EPI_PLAIN>()) != cudaSuccess) return e;
    if ((e = march_config<EPI_RESID>()) != cudaSuccess) return e;
    return march_config<EPI_CHEB>();
}

cudaError_t launch_march(int epi, const LevelGeom& g, const float* mu, const float* src, float* dst, const float* b,
                         const float* dinv, const float* d, float* d_new, double c1, double c2, cudaStream_t s) {
    if (epi == EPI_CHEB && (dst == src || d_new == d)) return cudaErrorInvalidValue;
    MarchArgs a{};
    a.n = g.n;
    a.M = g.M;
    a.oz = march_layers(g.n);
    a.nodes = g.nodes;
    a.h = float(g.h);
    a.mu = mu;
    a.src = src;
    a.dst = dst;
    a.b = b;
    a.dinv = dinv;
    a.d = d;
    a.d_new = d_new;
    a.c1 = float(c1);
    a.c2 = float(c2);
    const dim3 grid(unsigned((g.n + kTileX - 1) / kTileX), unsigned((g.n + kTileY - 1) / kTileY),
                    unsigned((g.n + a.oz - 1) / a.oz));
    if (epi == EPI_PLAIN)
        LAUNCH(PROF_VMULT_F32, s, (k_march<EPI_PLAIN><<<grid, kMarchThreads, sizeof(MarchShared<EPI_PLAIN>), s>>>(a)));
    else if (epi == EPI_RESID)
        LAUNCH(PROF_VMULT_F32, s, (k_march<EPI_RESID><<<grid, kMarchThreads, sizeof(MarchShared<EPI_RESID>), s>>>(a)));
    else
        LAUNCH(PROF_VMULT_F32, s, (k_march<EPI_CHEB><<<grid, kMarchThreads, sizeof(MarchShared<EPI_CHEB>), s>>>(a)));
    return cudaGetLastError();
}

}  // namespace stk
