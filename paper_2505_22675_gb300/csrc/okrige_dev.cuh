// Device code of local ordinary kriging (Sec. III-C) over the exact k nearest
// soundings, shared by the per-grid kernels (okrige.cu) and the batched
// persistent kernels (batch.cu).
//
// Per grid node: exact k-NN to neighbour ids (knn_warp.cuh, knn.cuh); then the
// kriging systems (okrige_solve_range).
//
// The bordered variogram system [Gamma 1; 1^T 0][lambda; mu] = [gamma_0; 1]
// is reduced with sum(lambda) = 1 by eliminating lambda_0 (the nearest
// neighbour) and mu. For reduced rows r, c (neighbours r+1, c+1):
//     A[r][c] = Gamma_r0 + Gamma_c0 - Gamma_rc,   b_r = Gamma_r0 + gamma_00 - gamma_r0,
//     A lambda' = b,  lambda_0 = 1 - sum(lambda'),  mu = gamma_00 - sum_a Gamma_0a lambda_a.
// A is symmetric positive definite for a conditionally negative definite
// variogram (spherical and exponential are, in 2-D), so |A[r][c]| is bounded
// by its largest diagonal entry.
//
// Layout: a warp's 32 lanes run 32 systems in step, so nothing is exchanged
// between lanes. Two threads share a system (one for K <= 8): the same lane of
// warps w and w + 4, each owning four rows of every tile; 8 warps per SM at
// K = 32, 16 at K = 16. The triangle is worked in tiles of 8 x 8 (left-looking
// block Cholesky): a tile is assembled from the rows' records into registers,
// updated with the factor's earlier columns, factored (by both threads alike,
// after an exchange through shared memory) or solved against the diagonal tile,
// and stored. The factor lives in tensor memory, used as a plain 128-lane store:
// lane l holds system l's 512 columns, exactly the 6 off-diagonal tiles of 64
// words and the 4 packed diagonal tiles of 28 (+ 4) of a K = 32 system, and both
// of its warps reach it. Shared memory could not hold it (2 KB x 128 systems
// + the records), and would serve one 128-byte wavefront per cycle to the
// whole SM where tensor memory serves each scheduler its own; the loads are
// issued four columns ahead of the multiplies. The records, right-hand sides
// and integer sums stay in shared memory, system-interleaved 16-byte vectors.
// The multiplies run as packed two-lane instructions (add/sub/mul/fma.rn.f32x2:
// one instruction, two IEEE single operations), two rows per instruction
// against one column's scalar in both lanes (which costs no extra
// instruction). The factor works on -A (the tile sums then need no negations).
// What bounds it: issue and latency at two warps per scheduler (half of the
// issue slots; FP32 pipe half busy in the factor, the square roots and
// conversions half busy in the residual), K = 32 with the fused IDW: 48,000
// cycles per 128 systems, of them factor 22,500, residual 11,300 (16,400 with the
// tiles evaluated again, 9,900 with them rounded to integers before they are
// kept, but then the factor takes 24,900), gathers 3,500.
// Measured on one survey line (3,001 x 692 nodes, k = 32, fused IDW): 2.52 ms
// (2.77 with the tiles evaluated again) against 3.84 ms for 8 threads per system
// with the factor in registers (1,500 warp instructions per system there, 664
// here; one thread per system: 630, but one warp per scheduler and 3.5 ms); 256 x
// 256 tile, k = 16: 28 against 37 us. Loading the next batch's ids and records
// during the last solve changed nothing.
//
// One step of iterative refinement follows the solve: A' is A rounded to a
// 30-bit fixed point, x is rounded to 24-bit fixed point x' (exact in FP32),
// and the residual b - A' x' is accumulated exactly in 64-bit integers. The
// tiles of A are kept for it: at K = 16 most of them in tensor memory beside
// the factor, at K = 32, where on-chip memory holds only one of the two
// triangles, in the threads' local memory (1.3 KB a thread, 50 MB over the
// device's resident systems: L2 holds them but for 0.4 KB a system that is
// written back, 6 % of the DRAM's bandwidth with the ids), read one tile ahead. CUDA
// takes 82 MB for it at the first launch, beside what the context counts.
// The correction reuses the factor. The weight sum closes in FP64: lambda_0 = 1 -
// sum(lambda'). Outputs:
//     zhat    = z_0 + sum_a lambda_a (z_a - z_0)          (= sum lambda_i z_i)
//     sigma^2 = lambda_0 gamma_00 + sum_a lambda_a gamma_a0 + mu.
// Rows beyond k_eff - 1 are identity rows with zero right-hand side, so every
// system has the fixed size K.
#pragma once

#include <algorithm>
#include <cmath>
#include <utility>

#include "bg_internal.h"
#include "idw_dev.cuh"
#include "knn.cuh"
#include "knn_warp.cuh"
#include "packed.cuh"

namespace bg {


constexpr int kSolveSystems = 128;  // systems per block, one lane of tensor memory each

template <int K>
struct Geo {
    static constexpr int TB = K < 8 ? K : 8;             // tile side
    static constexpr int NB = K / TB;                    // tile rows
    static constexpr int P = TB / 2;                     // row pairs of a tile
    static constexpr int TRI = TB * (TB - 1) / 2;        // strictly lower entries of a diagonal tile
    static constexpr int OFF = NB * (NB - 1) / 2;        // off-diagonal tiles
    static constexpr int TILE = TB * TB;                 // words of an off-diagonal tile
    static constexpr int DTILE = 32;                     // words of a packed diagonal tile
    static constexpr int TPS = NB > 1 ? 2 : 1;           // threads per system
    static constexpr int THREADS = TPS * kSolveSystems;
    // tensor-memory columns of a block (0: the factor stays in registers). At K =
    // 16 the two blocks of an SM have room for most of A' too: the off-diagonal
    // and the first diagonal tile, 32 words a thread each, from KEEP on.
    static constexpr int KEEP = OFF * TILE + NB * DTILE;
    static constexpr int COLS = NB == 1 ? 0 : K == 16 ? KEEP + 128 : KEEP;
    // shared memory, in 16-byte vectors per system: vectors of four rows
    static constexpr int Q = K / 4;
    static constexpr int X = 0, Y = Q, Z = 2 * Q;        // the rows' records
    static constexpr int DZ = 3 * Q, G0 = 4 * Q;         // z_a - z_0, gamma_0a
    static constexpr int V = 5 * Q;                      // L^-1 b, then x' (integers)
    static constexpr int DI = 6 * Q;                     // -1 / L[r][r]
    static constexpr int XB = 7 * Q;                     // exchange of eight rows, two buffers
    static constexpr int EX = XB + 4;                    // exchange of the prologue
    static constexpr int ACC = EX + 2;                   // 64-bit residual sums, one set a thread
    static constexpr int DG = ACC;                       // diagonal tile (16 vectors), before them
    static constexpr int VECS = NB == 1 ? ACC : ACC + 4 * Q;
    static constexpr int SMEM = VECS * 16 * kSolveSystems;
    // resident blocks per SM the registers are held to
    static constexpr int BLOCKS = K == 32 ? 1 : K == 16 ? 2 : 4;
};

__device__ __forceinline__ float variogram(const OkParams& p, float h_m) {
    if (p.model == BG_VARIOGRAM_SPHERICAL) {
        const float t = h_m * p.inv_a;
        if (t >= 1.0f) return p.sill;
        return fmaf(p.c * t, fmaf(-0.5f * t, t, 1.5f), p.c0);
    }
    // 1 - exp(-t) as -expm1(-t): no cancellation at short range, where the
    // model without a nugget makes the kriging variance small
    return fmaf(p.c, -expm1f(-h_m * p.inv_a), p.c0);
}

// gamma from a separation in cm; zero separation gives `at_zero`
__device__ __forceinline__ float gamma_cm(const OkParams& p, int dx, int dy, float at_zero) {
    if ((dx | dy) == 0) return at_zero;
    const float fx = (float)dx, fy = (float)dy;
    const float d2 = fmaf(fx, fx, fy * fy);
    return variogram(p, d2 * rsqrtf(d2) * 0.01f);
}

// one hardware square-root approximation (a few ulp, 0 at 0 and below 2^-126)
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 1 - exp(-t) for two t in [0, 25] at once (past 25 it is 1 in any case), for the
// exponential model: a solve is bound by its instructions, and two entries share
// each here, which a library call for each cannot (k = 12, 170,163 systems: solve
// 104 -> 75 us). Argument reduction of Cody and Waite: t = n ln 2 + r, |r| <= ln 2
// / 2; 1 - exp(-r) = r - r^2 q(r), q of degree 5 by interpolation at the Chebyshev
// nodes of that interval (off by 1.3e-9 at most); then (1 - s) + s (1 - exp(-r)), s
// = 2^-n, which does not cancel at short range. Errors, 2e6 draws in each of nine
// intervals: 0.89 ulp at most, 0.22 to 0.34 rms (-expm1f: 1.13, 0.22 to 0.50; with
// q of degree 4 1.01, 0.22 to 0.35 and 2 us less). Variances against 64 bits, relative rms
// error over 14 random tiles (k 8 to 32, ranges 20 to 76 m): 1.02e-7, with -expm1f 1.04e-7;
// of one tile between 0.83 and 1.04 times the latter.
__device__ __forceinline__ u64 one_minus_exp2(u64 t) {
    const u64 magic = dup2(12582912.0f);  // 1.5 * 2^23: the low bits of a sum hold the integer
    const u64 y = fma2(t, dup2(1.44269504f), magic);
    const u64 r = fma2(sub2(y, magic), dup2(-0.693147181f), t);
    u64 q = fma2(dup2(0.000198909911f), r, dup2(-0.00139336498f));
    q = fma2(q, r, dup2(0.00833331048f));
    q = fma2(q, r, dup2(-0.0416664667f));
    q = fma2(q, r, dup2(0.166666672f));
    q = fma2(q, r, dup2(-0.5f));
    const u64 m = fma2(mul2(r, r), q, r);
    const auto pow2 = [](float v) {  // 2^-n
        return __uint_as_float(0x3f800000u - (__float_as_uint(v) << 23));
    };
    const u64 s = pk2(pow2(lo2(y)), pow2(hi2(y)));
    return fma2(s, m, sub2(dup2(1.0f), s));
}
__device__ __forceinline__ float exp_clamp(float x, float most) {  // min that keeps a NaN
    float c;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(c) : "f"(x), "f"(most));
    return c;
}

// The variogram of the assembly in the fixed-point scale of the system: with
// the scale sa a power of two, sa gamma(h) is the model with c0 and c scaled
// by sa. t^2 = d2 (1/a)^2 from the exact squared separation in cm^2.
struct ScaledVgm {
    float kinv2;  // (0.01 / a)^2: cm^2 -> (h / a)^2
    float c0s;    // sa c0
    float cs;     // sa c
    float k2, k3; // spherical: -0.5 sa c, 1.5 sa c
};

__device__ __forceinline__ ScaledVgm scaled_vgm(const OkParams& p, float sa) {
    const float kinv = p.inv_a * 0.01f;
    const float cs = p.c * sa;
    return ScaledVgm{kinv * kinv, p.c0 * sa, cs, -0.5f * cs, 1.5f * cs};
}

// gamma between two distinct soundings from float offsets in cm (exact integers
// below 2^24), spherical model, for two rows at once (packed FP32); zero
// separation gives the nugget c0 (the h -> 0+ limit) without a branch: t =
// min(h / a, 1) makes the polynomial equal the sill beyond the range
__device__ __forceinline__ void gamma_pair_sph2(const OkParams& p, float dxa, float dya, float dxb,
                                                float dyb, float& ga, float& gb) {
    const unsigned long long dx = pk2(dxa, dxb), dy = pk2(dya, dyb);
    const unsigned long long d2 = fma2(dx, dx, mul2(dy, dy));
    float ea, eb;
    upk2(add2(d2, pk2(1e-30f, 1e-30f)), ea, eb);
    const unsigned long long h = mul2(d2, pk2(rsqrtf(ea), rsqrtf(eb)));
    float ta, tb;
    upk2(mul2(mul2(h, pk2(p.inv_a, p.inv_a)), pk2(0.01f, 0.01f)), ta, tb);
    const unsigned long long t = pk2(fminf(ta, 1.0f), fminf(tb, 1.0f));
    const unsigned long long in = fma2(mul2(pk2(-0.5f, -0.5f), t), t, pk2(1.5f, 1.5f));
    upk2(fma2(mul2(pk2(p.c, p.c), t), in, pk2(p.c0, p.c0)), ga, gb);
}

// gamma_cm (zero separation gives 0), spherical model, for two rows at once
__device__ __forceinline__ void gamma_cm_sph2(const OkParams& p, int dxa, int dya, int dxb, int dyb,
                                              float& ga, float& gb) {
    const unsigned long long fx = pk2((float)dxa, (float)dxb), fy = pk2((float)dya, (float)dyb);
    const unsigned long long d2 = fma2(fx, fx, mul2(fy, fy));
    float da, db;
    upk2(d2, da, db);
    float ta, tb;
    upk2(mul2(mul2(mul2(d2, pk2(rsqrtf(da), rsqrtf(db))), pk2(0.01f, 0.01f)), pk2(p.inv_a, p.inv_a)),
         ta, tb);
    const unsigned long long t = pk2(ta, tb);
    const unsigned long long in = fma2(mul2(pk2(-0.5f, -0.5f), t), t, pk2(1.5f, 1.5f));
    float va, vb;
    upk2(fma2(mul2(pk2(p.c, p.c), t), in, pk2(p.c0, p.c0)), va, vb);
    ga = ((dxa | dya) == 0) ? 0.0f : (ta >= 1.0f ? p.sill : va);
    gb = ((dxb | dyb) == 0) ? 0.0f : (tb >= 1.0f ? p.sill : vb);
}

// The two above, exponential model
__device__ __forceinline__ void gamma_pair_exp2(const OkParams& p, float dxa, float dya, float dxb, float dyb,
                                                float& ga, float& gb) {
    const u64 dx = pk2(dxa, dxb), dy = pk2(dya, dyb);
    const u64 d2 = fma2(dx, dx, mul2(dy, dy));
    const u64 e = add2(d2, dup2(1e-30f));
    float ta, tb;
    upk2(mul2(mul2(mul2(d2, pk2(rsqrtf(lo2(e)), rsqrtf(hi2(e)))), dup2(p.inv_a)), dup2(0.01f)), ta, tb);
    const u64 t = pk2(exp_clamp(ta, 25.0f), exp_clamp(tb, 25.0f));
    upk2(fma2(dup2(p.c), one_minus_exp2(t), dup2(p.c0)), ga, gb);
}
__device__ __forceinline__ void gamma_cm_exp2(const OkParams& p, int dxa, int dya, int dxb, int dyb,
                                              float& ga, float& gb) {
    const u64 fx = pk2((float)dxa, (float)dxb), fy = pk2((float)dya, (float)dyb);
    const u64 d2 = fma2(fx, fx, mul2(fy, fy));
    float ta, tb;
    upk2(mul2(mul2(mul2(d2, pk2(rsqrtf(lo2(d2)), rsqrtf(hi2(d2)))), dup2(0.01f)), dup2(p.inv_a)), ta, tb);
    const u64 t = pk2(exp_clamp(ta, 25.0f), exp_clamp(tb, 25.0f));
    float va, vb;
    upk2(fma2(dup2(p.c), one_minus_exp2(t), dup2(p.c0)), va, vb);
    ga = (dxa | dya) == 0 ? 0.0f : va;
    gb = (dxb | dyb) == 0 ? 0.0f : vb;
}

// ------------------------------------------------------------ k-NN -> ids

// The neighbour ids of a range of systems, in one of two layouts.
//   rows (stride 0): system i's k ids at p[i k], upload indices, -1 past k_eff;
//     system i is the i-th node (row-major) or point of the range.
//   patches (stride > 0): id n of system i at p[n stride + i], so that a warp's
//     loads and stores are whole lines; systems are the slots of 8 x 4 node
//     patches (32 per patch, patches row-major, the ones outside the grid
//     unused). A value >= 0 is a position in the cell-sorted records, whose
//     neighbours in space are neighbours in memory; -1 none; -2 - u the upload
//     index u (a node that the per-thread search served).
struct IdsView {
    int32_t* p;
    int64_t stride;
    int pnx;     // patches: per row of patches
    int j0, j1;  // patches: the range's grid rows
};
// Does the patches layout pay? The solve reads it in whole lines, but runs its unused
// slots like any other. k = 32, us, slots / rows: 1024 x 1024 nodes 1535 / 1692, 316 x
// 316 (1.3 % unused) 290 / 291, 14 x 10,000 (14 %) 285 / 280, 20 x 10,000 (20 %) 397
// / 379, 4 x 50,000 (half) 605 / 400; k = 16: 486 / 537, 136 / 136, 100 / 100, 130 /
// 127, 194 / 134.
__host__ __device__ inline bool slots_pay(int64_t slots, int64_t nodes) { return 10 * slots <= 11 * nodes; }
// grid node of a patch slot; false outside the grid
__device__ __forceinline__ bool slot_node(const IdsView& v, const GridView& g, int64_t slot, int& i, int& j) {
    const unsigned patch = (unsigned)(slot >> 5), py = patch / (unsigned)v.pnx;
    const int l = (int)(slot & 31);
    i = (int)(patch - py * (unsigned)v.pnx) * 8 + (l & 7);
    j = v.j0 + (int)py * 4 + (l >> 3);
    return i < g.nx && j < v.j1;
}
__device__ __forceinline__ int64_t node_slot(const IdsView& v, int i, int j) {
    return ((int64_t)((j - v.j0) >> 2) * v.pnx + (i >> 3)) * 32 + ((j - v.j0) & 3) * 8 + (i & 7);
}

// The k ids of a node that the patch search served, to slot `o` of the patches
// layout (or, with stride 0, to o[0 .. k) as upload indices).
template <int K>
__device__ __forceinline__ void ids_served(const HashView& h, const typename KnnWarp<K>::Smem& sm, int k, int32_t* o,
                                           int64_t stride) {
    const uint32_t* col = sm.buf + (threadIdx.x & 31);
    if (stride > 0) {
#pragma unroll 8
        for (int n = 0; n < k; ++n) o[n * stride] = sm.pos[col[n * 32] & kPlaceMask];
    } else {
        for (int n = 0; n < k; ++n) o[n] = __ldg(&h.rec[sm.pos[col[n * 32] & kPlaceMask]].w);
    }
}
// The same of a node that it did not serve, by a per-thread search.
template <int K>
__device__ __noinline__ KnnFar ids_lone(const HashView& h, int qx, int qy, uint64_t* hp, float ub, int k,
                                        int32_t* o, int64_t stride) {
    const int cnt = knn_lane<K>(h, qx, qy, hp, ub);
    const uint64_t mask = (1ull << h.idx_bits) - 1;
    if (cnt < 0) return KnnFar{cnt, 0.0f, 0.0f};
    for (int n = 0; n < k; ++n) {
        const int u = n < cnt ? (int)(hp[n * 32] & mask) : -1;
        if (stride > 0)
            o[n * stride] = u < 0 ? -1 : -2 - u;
        else
            o[n] = u;
    }
    return knn_far<K>(h, hp, cnt);
}

// Wide-key neighbour ids of one grid node whose table bound does not fit the
// packed key; other nodes return.
template <int K>
__device__ __forceinline__ void knn_ids_node_wide(const HashView& h, const GridView& g, int k, const IdsView& ids,
                                                  NodeIdx nd) {
    if (nd.i >= g.nx || nd.j >= ids.j1 || h.n_valid == 0) return;
    const int qx = g.x0 + nd.i * g.cell + g.cell / 2;
    const int qy = g.y0 + nd.j * g.cell + g.cell / 2;
    const Bound b = knn_bound<K>(h, qx, qy);
    if (packed_fits(h, b.tau0)) return;
    uint64_t d2[K];
    int id[K];
    const int keff = knn_scan_wide<K>(h, qx, qy, b, d2, id);
    if (ids.stride == 0) {
        int32_t* o = ids.p + ((int64_t)(nd.j - ids.j0) * g.nx + nd.i) * k;
#pragma unroll
        for (int i = 0; i < K; ++i)
            if (i < k) o[i] = i < keff ? id[i] : -1;
    } else {
        int32_t* o = ids.p + node_slot(ids, nd.i, nd.j);
#pragma unroll
        for (int i = 0; i < K; ++i)
            if (i < k) o[i * ids.stride] = i < keff ? -2 - id[i] : -1;
    }
}

// Neighbour i of a query point, upload index u (-1: none), to o: the first slot of
// its list with stride 0 (the caller's lists), else its slot of the patches layout,
// which the solve reads in whole lines (a line per lane otherwise: 209,715 points k =
// 32: solve 289 -> 282 us).
__device__ __forceinline__ void put_point_id(int32_t* o, int64_t stride, int i, int u) {
    if (stride > 0)
        o[i * stride] = u < 0 ? -1 : -2 - u;
    else
        o[i] = u;
}

// Wide-key neighbour ids of one query point whose table bound does not fit
// the packed key; other points return.
template <int K>
__device__ __forceinline__ void knn_ids_point_wide(const HashView& h, int qx, int qy, int k,
                                                   int32_t* __restrict__ o, int64_t stride) {
    if (!point_may_be_wide(h, qx, qy)) return;
    const Bound b = knn_bound<K>(h, qx, qy);
    if (packed_fits(h, b.tau0)) return;
    uint64_t d2[K];
    int id[K];
    const int keff = knn_scan_wide<K>(h, qx, qy, b, d2, id);
#pragma unroll
    for (int i = 0; i < K; ++i)
        if (i < k) put_point_id(o, stride, i, i < keff ? id[i] : -1);
}

// ---------------------------------------------------------------- solve

__device__ __forceinline__ u64 pk2u(uint32_t a, uint32_t b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ------------------------------------------------------------ tensor memory
// A warp reaches the quarter of the 128 lanes that its index modulo 4 names, so the
// two warps of a system (w and w + 4) share theirs; a thread reads and writes its
// lane's columns (32x32b). Loads are collected by tmem_wait_ld, which takes the
// loaded registers as operands so that no use of them moves above it.

__device__ __forceinline__ void tmem_ld16(uint32_t (&r)[16], uint32_t a) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(a));
}
__device__ __forceinline__ void tmem_st16(uint32_t a, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};" ::"r"(r[0]),
        "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(a));
}
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])::"memory");
}
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[16], uint32_t (&s)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(s[0]), "+r"(s[1]),
                   "+r"(s[2]), "+r"(s[3]), "+r"(s[4]), "+r"(s[5]), "+r"(s[6]), "+r"(s[7]),
                   "+r"(s[8]), "+r"(s[9]), "+r"(s[10]), "+r"(s[11]), "+r"(s[12]), "+r"(s[13]),
                   "+r"(s[14]), "+r"(s[15])::"memory");
}
// further registers of loads that a tmem_wait_ld before it has collected
__device__ __forceinline__ void tmem_use(uint32_t (&r)[16]) {
    asm volatile(""
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
}
__device__ __forceinline__ void tmem_wait_st() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Around a barrier that hands tensor memory from one warp to another: what the one has
// read or written (and waited for) lies before what the other does with it.
__device__ __forceinline__ void tmem_before_sync() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_after_sync() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// A block's tensor memory (Geo<K>::COLS columns, a power of two), taken by warp
// 0 at the start and given back by it at the end; `slot` is a shared word.
// Returns the thread's base address (its warp's lanes).
template <int COLS>
__device__ __forceinline__ uint32_t tmem_take(uint32_t* slot) {
    if constexpr (COLS == 0) return 0;
    static_assert(COLS == 0 || COLS == 256 || COLS == 512, "an allocation size");
    if (threadIdx.x < 32) {
        const uint32_t sa = (uint32_t)__cvta_generic_to_shared(slot);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa),
                     "r"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tmem_before_sync();
    __syncthreads();
    tmem_after_sync();
    return *(volatile uint32_t*)slot + ((uint32_t)(threadIdx.x >> 5 & 3) << 21);
}
template <int COLS>
__device__ __forceinline__ void tmem_give(const uint32_t* slot) {
    if constexpr (COLS != 0) {
        tmem_before_sync();
        __syncthreads();
        tmem_after_sync();
        if (threadIdx.x < 32)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*slot),
                         "r"(COLS)
                         : "memory");
    }
}

// L2 prefetch of the neighbour ids of solve block pb of a range of `nsys`
// systems. A hint that nothing waits on.
__device__ __forceinline__ void prefetch_ids_l2(const IdsView& v, int64_t nsys, int k, int64_t pb) {
    const int t = threadIdx.x;
    const int64_t sys = pb * kSolveSystems;
    if (v.stride == 0) {
        if (t < kSolveSystems && sys + t < nsys)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(v.p + (sys + t) * k));
    } else if (sys < nsys) {
        for (int q = t; q < 4 * k; q += blockDim.x)  // 128 systems: four lines per neighbour
            if (sys + (q & 3) * 32 < nsys) asm volatile("prefetch.global.L2 [%0];" ::"l"(v.p + (q >> 2) * v.stride + sys + (q & 3) * 32));
    }
}

// 2^e as a float (|e| <= 126)
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

// exponent e with 2^(e-1) <= v < 2^e for finite v > 0
__device__ __forceinline__ int exp_above(float v) { return ((__float_as_int(v) >> 23) & 0xff) - 126; }

// round to nearest as int64 of |f| < 2^62, through two 32-bit conversions (a
// 64-bit one runs at the FP64 rate)
__device__ __forceinline__ long long float_to_ll(float f) {
    const int hi = __float2int_rn(f * 2.3283064365386963e-10f);     // 2^-32
    const int lo = __float2int_rn(fmaf((float)hi, -4294967296.0f, f));  // exact remainder
    return ((long long)hi << 32) + lo;
}
// the float nearest to v up to one rounding of its upper half
__device__ __forceinline__ float ll_to_float(long long v) {
    const int lo = (int)v;
    const int hi = (int)((v - lo) >> 32);
    return fmaf((float)hi, 4294967296.0f, (float)lo);
}

// The tile function of the assembly: -A for two rows at once, in the
// fixed-point scale. -A[r][c] = gamma(r, c) - Gamma_r0 - Gamma_c0; the records
// hold zr = -Gamma_r0, and zc comes in as c0 - Gamma_c0 (all scaled).
template <bool kSph>
struct TileVgm {
    u64 kinv2, k2, k3;
    float c0s, cs;
    __device__ __forceinline__ explicit TileVgm(const ScaledVgm& v)
        : kinv2(dup2(v.kinv2)), k2(dup2(v.k2)), k3(dup2(v.k3)), c0s(v.c0s), cs(v.cs) {}
    // (h / a)^2; an entry from it. A tile takes these one after the other for all
    // its entries: the chain of one entry (a square root in it) is far longer
    // than its issue slots.
    __device__ __forceinline__ u64 dist(u64 xr, u64 yr, float xc, float yc) const {
        const u64 dx = sub2(xr, dup2(xc)), dy = sub2(yr, dup2(yc));
        return mul2(fma2(dx, dx, mul2(dy, dy)), kinv2);
    }
    __device__ __forceinline__ u64 entry(u64 t2, u64 zr, float zc) const {
        float ta, tb;
        upk2(t2, ta, tb);
        if constexpr (kSph) {
            // the polynomial is the sill at t = 1
            ta = fminf(ta, 1.0f);
            tb = fminf(tb, 1.0f);
            const u64 in = fma2(k2, pk2(ta, tb), k3);
            return fma2(pk2(sqrt_approx(ta), sqrt_approx(tb)), in, add2(zr, dup2(zc)));
        } else {
            const u64 t = pk2(sqrt_approx(exp_clamp(ta, 625.0f)), sqrt_approx(exp_clamp(tb, 625.0f)));
            return fma2(dup2(cs), one_minus_exp2(t), add2(zr, dup2(zc)));
        }
    }
};

// Vectors of four rows of a system (see Geo): load / store the TB rows of tile
// row b of array `at`.
template <int K>
struct Lane {
    using Gm = Geo<K>;
    static constexpr int TB = Gm::TB, P = Gm::P;
    float4* s;  // the system's vectors, kSolveSystems apart
    __device__ __forceinline__ float4& vec(int i) const { return s[i * kSolveSystems]; }
    // rows 2 p, 2 p + 1 of tile row b
    __device__ __forceinline__ float2& pair(int at, int b, int p) const {
        return reinterpret_cast<float2*>(&vec(at + b * (TB / 4) + (p >> 1)))[p & 1];
    }
    __device__ __forceinline__ longlong2& long2(int at) const {
        return *reinterpret_cast<longlong2*>(&vec(at));
    }
    __device__ __forceinline__ void pairs(int at, int b, u64 (&p)[P]) const {
#pragma unroll
        for (int i = 0; i < TB / 4; ++i) {
            const float4 f = vec(at + b * (TB / 4) + i);
            p[2 * i] = pk2(f.x, f.y);
            p[2 * i + 1] = pk2(f.z, f.w);
        }
    }
    __device__ __forceinline__ void floats(int at, int b, float (&p)[TB]) const {
#pragma unroll
        for (int i = 0; i < TB / 4; ++i) {
            const float4 f = vec(at + b * (TB / 4) + i);
            p[4 * i] = f.x;
            p[4 * i + 1] = f.y;
            p[4 * i + 2] = f.z;
            p[4 * i + 3] = f.w;
        }
    }
    __device__ __forceinline__ void put(int at, int b, const float (&p)[TB]) const {
#pragma unroll
        for (int i = 0; i < TB / 4; ++i)
            vec(at + b * (TB / 4) + i) =
                make_float4(p[4 * i], p[4 * i + 1], p[4 * i + 2], p[4 * i + 3]);
    }
    __device__ __forceinline__ void ints(int at, int b, int (&p)[TB]) const {
        float f[TB];
        floats(at, b, f);
#pragma unroll
        for (int i = 0; i < TB; ++i) p[i] = __float_as_int(f[i]);
    }
    __device__ __forceinline__ void put_ints(int at, int b, const int (&p)[TB]) const {
        float f[TB];
#pragma unroll
        for (int i = 0; i < TB; ++i) f[i] = __int_as_float(p[i]);
        put(at, b, f);
    }
};

// With two threads per system, thread h of a system owns row pairs p = h and
// 3 - h of every tile (rows 0, 1, 6, 7 or 2, 3, 4, 5: equal shares of the
// diagonal tiles too), so the multiplies of a tile split without exchange; an
// off-diagonal tile of the factor is stored as two halves of 32 words, the
// four owned rows of column c at 4 c. The two threads of a system sit in
// warps w and w + 4 (the same lanes of tensor memory) and meet at a named
// barrier of the two warps.
__device__ __forceinline__ void pair_sync() {
    asm volatile("bar.sync %0, 64;" ::"r"(1 + (int)(threadIdx.x >> 5 & 3)) : "memory");
}
// tensor memory that one warp of the pair has read (the loads waited for) or written
// is the other's to write or read
__device__ __forceinline__ void pair_sync_tmem() {
    tmem_wait_st();
    tmem_before_sync();
    pair_sync();
    tmem_after_sync();
}
// row r of a tile as (half, place): the half that owns it and its place there
constexpr __host__ __device__ int half_of(int r) { return r >= 2 && r < 6; }
constexpr __host__ __device__ int place_of(int r) { return r < 2 ? r : r < 6 ? r - 2 : r - 4; }

// Row pairs p[0], p[1] (tile row I) of -A's tile columns: t[u][c] is pair
// p[u] of column c of tile (I, J). Rows past the last neighbour have no
// coupling (off-diagonal zero); full: every neighbour of the warp's systems real.
template <int K, bool kSph>
__device__ __forceinline__ void assemble_off(const Lane<K>& ln, const TileVgm<kSph>& vg, int I,
                                             int J, const int (&pr)[2], int ke, bool full,
                                             u64 (&t)[2][8]) {
    using Gm = Geo<K>;
    u64 xr[2], yr[2], zr[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const float2 a = ln.pair(Gm::X, I, pr[u]), b = ln.pair(Gm::Y, I, pr[u]),
                     c = ln.pair(Gm::Z, I, pr[u]);
        xr[u] = pk2(a.x, a.y);
        yr[u] = pk2(b.x, b.y);
        zr[u] = pk2(c.x, c.y);
    }
    float xc[8], yc[8], zc[8];
    ln.floats(Gm::X, J, xc);
    ln.floats(Gm::Y, J, yc);
    ln.floats(Gm::Z, J, zc);
#pragma unroll
    for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int u = 0; u < 2; ++u) t[u][c] = vg.dist(xr[u], yr[u], xc[c], yc[c]);
#pragma unroll
    for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int u = 0; u < 2; ++u) t[u][c] = vg.entry(t[u][c], zr[u], zc[c] + vg.c0s);
    if (!full) {
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                float a, b;
                upk2(t[u][c], a, b);
                const int r = I * 8 + 2 * pr[u];
                t[u][c] = pk2(r + 1 < ke ? a : 0.0f, r + 2 < ke ? b : 0.0f);
            }
    } else if (I + 1 == Gm::NB && pr[1] == 3) {  // a whole system lacks only its last row
#pragma unroll
        for (int c = 0; c < 8; ++c) t[1][c] = pk2(lo2(t[1][c]), 0.0f);
    }
}

// Row pair p of -A's diagonal tile J, columns 0 .. 2 p + 1 (the entry above the
// diagonal is not used); on the diagonal of rows past the last neighbour the
// identity in the fixed-point scale.
template <int K, bool kSph, int p>
__device__ __forceinline__ void assemble_diag(const Lane<K>& ln, const TileVgm<kSph>& vg, int J, int ke, float sa,
                                              bool full, const float (&xc)[8], const float (&yc)[8],
                                              const float (&zc)[8], u64 (&t)[2 * p + 2]) {
    const u64 xr = pk2(xc[2 * p], xc[2 * p + 1]), yr = pk2(yc[2 * p], yc[2 * p + 1]),
              zr = pk2(zc[2 * p], zc[2 * p + 1]);
#pragma unroll
    for (int c = 0; c < 2 * p + 2; ++c) t[c] = vg.dist(xr, yr, xc[c], yc[c]);
#pragma unroll
    for (int c = 0; c < 2 * p + 2; ++c) t[c] = vg.entry(t[c], zr, zc[c] + vg.c0s);
    // -A[c][c] = -2 Gamma_c0
    float d0 = 2.0f * zc[2 * p], d1 = 2.0f * zc[2 * p + 1];
    if (!full) {
        const int r = J * 8 + 2 * p;
        const bool real0 = r + 1 < ke, real1 = r + 2 < ke;
        d0 = real0 ? d0 : -sa;
        d1 = real1 ? d1 : -sa;
#pragma unroll
        for (int c = 0; c < 2 * p + 2; ++c) t[c] = pk2(real0 ? lo2(t[c]) : 0.0f, real1 ? hi2(t[c]) : 0.0f);
    } else if (p == 3 && J + 1 == Geo<K>::NB) {  // a whole system lacks only its last row
        d1 = -sa;
#pragma unroll
        for (int c = 0; c < 2 * p + 2; ++c) t[c] = pk2(lo2(t[c]), 0.0f);
    }
    t[2 * p] = pk2(d0, hi2(t[2 * p]));
    t[2 * p + 1] = pk2(lo2(t[2 * p + 1]), d1);
}

// The whole -A of a one-tile system: t[c][p], the pairs that hold a row >= c
template <int K, bool kSph>
__device__ __forceinline__ void assemble_one(const Lane<K>& ln, const TileVgm<kSph>& vg, int ke,
                                             float sa, u64 (&t)[Geo<K>::TB][Geo<K>::P]) {
    using Gm = Geo<K>;
    u64 xr[Gm::P], yr[Gm::P], zr[Gm::P];
    ln.pairs(Gm::X, 0, xr);
    ln.pairs(Gm::Y, 0, yr);
    ln.pairs(Gm::Z, 0, zr);
#pragma unroll
    for (int c = 0; c < Gm::TB; ++c) {
        const float z0 = lane2(zr[c / 2], c & 1);
        const float z = z0 + vg.c0s;
#pragma unroll
        for (int p = c / 2; p < Gm::P; ++p) {
            float a, b;
            upk2(vg.entry(vg.dist(xr[p], yr[p], lane2(xr[c / 2], c & 1), lane2(yr[c / 2], c & 1)), zr[p], z), a, b);
            t[c][p] = pk2(2 * p + 1 < ke ? a : 0.0f, 2 * p + 2 < ke ? b : 0.0f);
        }
        const float d = c + 1 < ke ? 2.0f * z0 : -sa;  // -A[c][c] = -2 Gamma_c0
        t[c][c / 2] = (c & 1) ? pk2(lo2(t[c][c / 2]), d) : pk2(d, hi2(t[c][c / 2]));
    }
}

// Factor a diagonal tile t[c][p] of -A (less the earlier columns) in
// registers: the strictly lower entries column after column, ni = -1 /
// diagonal, and one step of L y = v on the tile's rows (nvp = -v in, y out).
template <int TB>
__device__ __forceinline__ void factor_tile(u64 (&t)[TB][TB / 2], u64 (&nvp)[TB / 2],
                                            float (&Ld)[TB * (TB - 1) / 2], float (&ni)[TB],
                                            float (&y)[TB]) {
    constexpr int P = TB / 2;
    int at = 0;
#pragma unroll
    for (int c = 0; c < TB; ++c) {
        ni[c] = -rsqrt_approx(-lane2(t[c][c / 2], c & 1));
        const u64 m = dup2(ni[c]);
        u64 L[P];
#pragma unroll
        for (int q = 0; q < P; ++q)
            if (2 * q + 1 > c) L[q] = mul2(t[c][q], m);
        y[c] = lane2(nvp[c / 2], c & 1) * ni[c];
#pragma unroll
        for (int r = c + 1; r < TB; ++r) {
            const float l = lane2(L[r / 2], r & 1);
            Ld[at++] = l;
#pragma unroll
            for (int q = r / 2; q < P; ++q) t[r][q] = fma2(L[q], dup2(l), t[r][q]);
        }
#pragma unroll
        for (int q = 0; q < P; ++q)
            if (2 * q + 1 > c) nvp[q] = fma2(L[q], dup2(y[c]), nvp[q]);
    }
}

// forward substitution with a diagonal tile: nv = -v in, y out (L y = v)
template <int TB>
__device__ __forceinline__ void diag_forward(const float (&Ld)[TB * (TB - 1) / 2],
                                             const float (&ni)[TB], float (&nv)[TB]) {
    int at = 0;
#pragma unroll
    for (int c = 0; c < TB; ++c) {
        nv[c] *= ni[c];
#pragma unroll
        for (int r = c + 1; r < TB; ++r) nv[r] = fmaf(Ld[at++], nv[c], nv[r]);
    }
}
// back substitution: nv = -v in, x out (L^T x = v)
template <int TB>
__device__ __forceinline__ void diag_backward(const float (&Ld)[TB * (TB - 1) / 2],
                                              const float (&ni)[TB], float (&nv)[TB]) {
#pragma unroll
    for (int c = TB - 1; c >= 0; --c) {
        nv[c] *= ni[c];
#pragma unroll
        for (int j = 0; j < c; ++j)  // L[c][j] in column-major order below the diagonal
            nv[j] = fmaf(Ld[j * TB - j * (j + 1) / 2 + (c - j - 1)], nv[c], nv[j]);
    }
}

// The kriging systems of batches b0 .. b1 - 1 (128 systems each) of a range of
// nsys, with the neighbour ids of `ids`; node0: the range's first node (rows
// layout). smem: Geo<K>::SMEM bytes; tm: the thread's tensor memory. With kPts
// the systems are query points whose coordinates are px[], py[] (g unused).
// With kIdw the block also writes the IDW depth over the first fz.k of the
// node's sorted neighbours (fz.k <= k): the same value bg_interp_idw gives, as
// its operations are those of idw_sum in the same order. Every warp reaches
// every barrier and tensor-memory instruction (idle lanes run the tile loops
// too).
template <int K, bool kSph, bool kPts, bool kIdw>
__device__ __forceinline__ void okrige_solve_range(const HashView& h, const GridView& g, int k,
                                                   const OkParams& p, int64_t node0, int64_t nsys,
                                                   const IdsView& ids,
                                                   float* __restrict__ depth,
                                                   float* __restrict__ var, int64_t b0, int64_t b1,
                                                   float4* smem, uint32_t tm,
                                                   const int32_t* __restrict__ px = nullptr,
                                                   const int32_t* __restrict__ py = nullptr,
                                                   IdwFuse fz = IdwFuse{}) {
    using Gm = Geo<K>;
    constexpr int TB = Gm::TB, NB = Gm::NB, P = Gm::P, TPS = Gm::TPS;
    const int lane = threadIdx.x % kSolveSystems;
    const int hh = TPS == 2 ? (int)threadIdx.x / kSolveSystems : 0;  // which thread of the system
    const Lane<K> ln{smem + lane};
#pragma unroll 1
    for (int64_t blk = b0; blk < b1; ++blk) {
    const int64_t sys = blk * kSolveSystems + lane;
    bool live = sys < nsys;
    int64_t node = node0 + (live ? sys : 0);
    int qx, qy;
    if constexpr (kPts) {
        qx = __ldg(px + node);
        qy = __ldg(py + node);
    } else {
        int i, j;
        if (ids.stride > 0) {
            live = slot_node(ids, g, live ? sys : 0, i, j) && live;
            node = (int64_t)j * g.nx + i;
        } else if (node < ((int64_t)1 << 31)) {
            j = (int)((unsigned)node / (unsigned)g.nx);
            i = (int)((unsigned)node - (unsigned)j * (unsigned)g.nx);
        } else {
            j = (int)(node / g.nx);
            i = (int)(node % g.nx);
        }
        qx = g.x0 + i * g.cell + g.cell / 2;
        qy = g.y0 + j * g.cell + g.cell / 2;
    }

    // ---- the neighbours: ids (-1 exactly past k_eff), records, variograms.
    // Thread hh takes the groups of four neighbours 4 q + 1 .. 4 q + 4 (reduced
    // rows 4 q .. 4 q + 3) with q = hh mod TPS; every load is issued before the
    // first use.
    constexpr int NQ = K / 4 / TPS;
    int nid[4 * NQ], id0;
    {
        const int32_t* my = ids.p + (live ? sys : 0) * (ids.stride > 0 ? 1 : k);
        const int64_t step = ids.stride > 0 ? ids.stride : 1;
        id0 = live ? __ldg(my) : -1;
#pragma unroll
        for (int i = 0; i < 4 * NQ; ++i) {
            const int n = 4 * (TPS * (i / 4) + hh) + i % 4 + 1;
            nid[i] = (live && n < k) ? __ldg(my + n * step) : -1;
        }
    }
    // positions come from the records, upload indices from the upload order
    const int4* const pos_base = ids.stride > 0 ? h.rec : h.orig;
    auto record = [&](int id) {
        return id >= 0 ? __ldg(pos_base + id) : id < -1 ? __ldg(h.orig + (-2 - id)) : make_int4(0, 0, 0, 0);
    };
    const int4 r0 = record(id0);
    int4 rr[4 * NQ];
    int ke = 0;
#pragma unroll
    for (int i = 0; i < 4 * NQ; ++i) {
        rr[i] = record(nid[i]);
        ke += nid[i] != -1 ? 1 : 0;
    }
    const float z0 = __int_as_float(r0.z);
    const float g00 = gamma_cm(p, r0.x - qx, r0.y - qy, 0.0f);
    float gr0[4 * NQ];  // Gamma(row's neighbour, neighbour 0)
    float gmax = 0.0f;
    bool idw_on = false;  // the node lies on a sounding
    float idw_num = 0.0f, idw_den = 0.0f;
    if constexpr (kIdw) {
        // idw_from's terms, in its order and partials: thread hh holds the partials
        // 4 hh .. 4 hh + 3 of neighbours n >= 1 (n - 1 = 4 q + u, q = hh mod 2)
        static_assert(TPS == 2 && kIdwLanes == 8, "the fused IDW runs with 2 threads per system");
        // (32-bit distances where they fit in the whole warp: the same floats)
        constexpr int kNear = 32000;
        bool near = id0 == -1 || (abs(r0.x - qx) < kNear && abs(r0.y - qy) < kNear);
        int ax[4 * NQ], ay[4 * NQ];
#pragma unroll
        for (int i = 0; i < 4 * NQ; ++i) {
            ax[i] = rr[i].x - qx;
            ay[i] = rr[i].y - qy;
            near &= nid[i] == -1 || (abs(ax[i]) < kNear && abs(ay[i]) < kNear);
        }
        float d[4 * NQ], d1;
        if (__all_sync(kFull, near)) {
            d1 = __int2float_rn((r0.x - qx) * (r0.x - qx) + (r0.y - qy) * (r0.y - qy));
#pragma unroll
            for (int i = 0; i < 4 * NQ; ++i) d[i] = __int2float_rn(ax[i] * ax[i] + ay[i] * ay[i]);
        } else {
            auto far = [&](int x, int y) {
                const long long dx = (long long)x - qx, dy = (long long)y - qy;
                return idw_d2f((uint64_t)(dx * dx + dy * dy));
            };
            d1 = far(r0.x, r0.y);
#pragma unroll 1
            for (int i = 0; i < 4 * NQ; ++i) {
                int x = 0, y = 0;
#pragma unroll
                for (int e = 0; e < 4 * NQ; ++e) {
                    x = e == i ? rr[e].x : x;
                    y = e == i ? rr[e].y : y;
                }
                const float v = far(x, y);
#pragma unroll
                for (int e = 0; e < 4 * NQ; ++e) d[e] = e == i ? v : d[e];
            }
        }
        idw_on = d1 == 0.0f;
        float num[4], den[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) num[u] = den[u] = 0.0f;
        auto terms = [&](float l1, float power) {
#pragma unroll
            for (int i = 0; i < 4 * NQ; ++i) {
                const int n = 4 * (2 * (i / 4) + hh) + i % 4 + 1;
                if (n >= fz.k) break;  // uniform over the warp
                const float w = idw_weight(d1, l1, 0.5f * power, power, d[i]);
                if (nid[i] != -1) {
                    num[i % 4] = fmaf(w, __int_as_float(rr[i].z) - z0, num[i % 4]);
                    den[i % 4] += w;
                }
            }
        };
        if (fz.power == 2.0f)
            terms(0.0f, 2.0f);
        else
            terms(log2f(d1), fz.power);
        idw_num = (num[0] + num[1]) + (num[2] + num[3]);
        idw_den = (den[0] + den[1]) + (den[2] + den[3]);
    }
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        const int q = TPS * j + hh;
        float ox[4], oy[4], dz[4], g0[4];
        int pdx[4], pdy[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int4 v = rr[4 * j + u];
            const bool real = nid[4 * j + u] != -1;
            ox[u] = real ? (float)(v.x - r0.x) : 0.0f;
            oy[u] = real ? (float)(v.y - r0.y) : 0.0f;
            dz[u] = real ? __int_as_float(v.z) - z0 : 0.0f;
            pdx[u] = v.x - qx;
            pdy[u] = v.y - qy;
        }
        if constexpr (kSph) {
#pragma unroll
            for (int u = 0; u < 4; u += 2) {
                gamma_pair_sph2(p, ox[u], oy[u], ox[u + 1], oy[u + 1], gr0[4 * j + u],
                                gr0[4 * j + u + 1]);
                gamma_cm_sph2(p, pdx[u], pdy[u], pdx[u + 1], pdy[u + 1], g0[u], g0[u + 1]);
            }
        } else {
#pragma unroll
            for (int u = 0; u < 4; u += 2) {
                gamma_pair_exp2(p, ox[u], oy[u], ox[u + 1], oy[u + 1], gr0[4 * j + u], gr0[4 * j + u + 1]);
                gamma_cm_exp2(p, pdx[u], pdy[u], pdx[u + 1], pdy[u + 1], g0[u], g0[u + 1]);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (nid[4 * j + u] == -1) gr0[4 * j + u] = g0[u] = 0.0f;
            gmax = fmaxf(gmax, gr0[4 * j + u]);
        }
        ln.vec(Gm::X + q) = make_float4(ox[0], ox[1], ox[2], ox[3]);
        ln.vec(Gm::Y + q) = make_float4(oy[0], oy[1], oy[2], oy[3]);
        ln.vec(Gm::DZ + q) = make_float4(dz[0], dz[1], dz[2], dz[3]);
        ln.vec(Gm::G0 + q) = make_float4(g0[0], g0[1], g0[2], g0[3]);
    }
    if constexpr (TPS == 2) {
        ln.vec(Gm::EX + hh) = make_float4(gmax, __int_as_float(ke), idw_num, idw_den);
        pair_sync();
        const float4 o = ln.vec(Gm::EX + 1 - hh);
        gmax = fmaxf(gmax, o.x);
        ke += __float_as_int(o.y);
        idw_num += o.z;
        idw_den += o.w;
    }
    ke = id0 != -1 ? ke + 1 : 0;  // neighbours; 0: no output (no data, or past the end)
    if constexpr (kIdw) {
        if (live && hh == 0)
            fz.out[node] = ke == 0 ? __int_as_float(0x7fc00000)
                                   : (idw_on ? z0 : z0 + idw_num / (1.0f + idw_den));
    }
    // A is SPD, so |A[r][c]| <= its largest diagonal entry max(1, 2 max Gamma_r0);
    // fixed point with 30 bits below that bound
    const int ea = 30 - exp_above(fmaxf(1.0f, 2.0f * gmax));
    const float sa = pow2f(ea), isa = pow2f(-ea);
#pragma unroll
    for (int j = 0; j < NQ; ++j)
        ln.vec(Gm::Z + TPS * j + hh) = make_float4(-gr0[4 * j] * sa, -gr0[4 * j + 1] * sa,
                                                   -gr0[4 * j + 2] * sa, -gr0[4 * j + 3] * sa);
    const TileVgm<kSph> vg(scaled_vgm(p, sa));
    // -b in the scale, of row r with records z = -sa Gamma_r0 and g0 = gamma_0r
    auto minus_b = [&](int r, float z, float g0) {
        return r + 1 < ke ? -(__fadd_rn(__fadd_rn(-z * isa, g00), -g0) * sa) : 0.0f;
    };

    if constexpr (NB == 1) {
        // ---- one tile: everything of the solve in registers
        float nv[TB], ni[TB], Ld[Gm::TRI], b[TB];
        {
            float z[TB], g0[TB];
            ln.floats(Gm::Z, 0, z);
            ln.floats(Gm::G0, 0, g0);
#pragma unroll
            for (int r = 0; r < TB; ++r) b[r] = minus_b(r, z[r], g0[r]);
        }
        u64 t[TB][P];
        {
            u64 nvp[P];
#pragma unroll
            for (int q = 0; q < P; ++q) nvp[q] = pk2(b[2 * q], b[2 * q + 1]);
            assemble_one<K, kSph>(ln, vg, ke, sa, t);
            factor_tile<TB>(t, nvp, Ld, ni, nv);
        }
#pragma unroll
        for (int r = 0; r < TB; ++r) nv[r] = -nv[r];
        diag_backward<TB>(Ld, ni, nv);
        float xmax = 0.0f;
#pragma unroll
        for (int r = 0; r < TB; ++r) xmax = fmaxf(xmax, fabsf(nv[r]));
        const int ex = xmax > 0.0f ? 24 - exp_above(xmax) : 0;
        const float sx = pow2f(ex), isx = pow2f(-ex);
        int xq[TB];
        long long acc[TB];
#pragma unroll
        for (int r = 0; r < TB; ++r) {
            xq[r] = __float2int_rn(nv[r] * sx);
            acc[r] = float_to_ll(-b[r] * sx);
        }
        assemble_one<K, kSph>(ln, vg, ke, sa, t);
#pragma unroll
        for (int c = 0; c < TB; ++c)
#pragma unroll
            for (int r = c; r < TB; ++r) {
                const int a = __float2int_rn(lane2(t[c][r / 2], r & 1));
                acc[r] += (long long)a * xq[c];
                if (r != c) acc[c] += (long long)a * xq[r];
            }
#pragma unroll
        for (int r = 0; r < TB; ++r) nv[r] = -(ll_to_float(acc[r]) * isx);  // -sa (b - A' x')
        diag_forward<TB>(Ld, ni, nv);
#pragma unroll
        for (int r = 0; r < TB; ++r) nv[r] = -nv[r];
        diag_backward<TB>(Ld, ni, nv);
        int sq = 0;
        float ps = 0.0f, pz = 0.0f, pv = 0.0f, dz[TB], g0[TB], z[TB];
        ln.floats(Gm::DZ, 0, dz);
        ln.floats(Gm::G0, 0, g0);
        ln.floats(Gm::Z, 0, z);
#pragma unroll
        for (int r = 0; r < TB; ++r) {
            const float lam = __fadd_rn(__fmul_rn((float)xq[r], isx), nv[r]);
            sq += xq[r];
            ps = __fadd_rn(ps, nv[r]);
            pz = fmaf(lam, dz[r], pz);                            // z_a - z_0
            pv = fmaf(lam, __fadd_rn(g0[r], z[r] * isa), pv);     // gamma_0a - Gamma_a0
        }
        const float lam0 = (float)(1.0 - ((double)sq * (double)isx + (double)ps));
        if (live) {
            if (ke == 0) {
                depth[node] = __int_as_float(0x7fc00000);  // no valid sounding
                if (var) var[node] = __int_as_float(0x7fc00000);
            } else {
                depth[node] = z0 + pz;
                if (var) var[node] = fmaf(lam0, g00, g00 + pv);
            }
        }
    } else {
        pair_sync();  // every record is there
        // every row but the last (row K - 1 has no neighbour) real, in the whole warp
        const bool full = __all_sync(kFull, ke == K);
        const int pr[2] = {hh, 3 - hh};  // owned row pairs
        const auto tcol = [&](int I, int J) {  // off-diagonal tile (I, J)
            return tm + (uint32_t)((I * (I - 1) / 2 + J) * Gm::TILE);
        };
        const auto dcol = [&](int J) { return tm + (uint32_t)(Gm::OFF * Gm::TILE + J * Gm::DTILE); };
        float Ld[Gm::TRI], ni[TB];  // the diagonal tile at hand and -1 / its diagonal
        float4 kept[K == 32 ? 8 * (NB * (NB + 1) / 2) : 1];  // K = 32: -A of this thread's rows, tile (I, J) at 8 (I (I + 1) / 2 + J)

        // ---- factor -A tile column by tile column; L y = b along the way
#pragma unroll 1
        for (int J = 0; J < NB; ++J) {
            // (each thread of the pair its own code: pairs 0 and 3 or 1 and 2)
            auto diag_part = [&](auto which) {
                constexpr int p0 = decltype(which)::value, p1 = 3 - p0, N0 = 2 * p0 + 2, N1 = 2 * p1 + 2;
                u64 t0[N0], t1[N1], nv[2];
                {
                    float xc[8], yc[8], zc[8], g0[8];
                    ln.floats(Gm::X, J, xc);
                    ln.floats(Gm::Y, J, yc);
                    ln.floats(Gm::Z, J, zc);
                    ln.floats(Gm::G0, J, g0);
                    assemble_diag<K, kSph, p0>(ln, vg, J, ke, sa, full, xc, yc, zc, t0);
                    assemble_diag<K, kSph, p1>(ln, vg, J, ke, sa, full, xc, yc, zc, t1);
                    nv[0] = pk2(minus_b(8 * J + 2 * p0, zc[2 * p0], g0[2 * p0]),
                                minus_b(8 * J + 2 * p0 + 1, zc[2 * p0 + 1], g0[2 * p0 + 1]));
                    nv[1] = pk2(minus_b(8 * J + 2 * p1, zc[2 * p1], g0[2 * p1]),
                                minus_b(8 * J + 2 * p1 + 1, zc[2 * p1 + 1], g0[2 * p1 + 1]));
                }
                if (K == 16 && J == 0) {  // kept for the residual: a = -A' of the first diagonal tile
                    uint32_t w[32];
#pragma unroll
                    for (int c = 0; c < N0; ++c) {
                        w[2 * c] = (uint32_t)__float2int_rn(lo2(t0[c]));
                        w[2 * c + 1] = (uint32_t)__float2int_rn(hi2(t0[c]));
                    }
#pragma unroll
                    for (int c = 0; c < N1; ++c) {
                        w[2 * (N0 + c)] = (uint32_t)__float2int_rn(lo2(t1[c]));
                        w[2 * (N0 + c) + 1] = (uint32_t)__float2int_rn(hi2(t1[c]));
                    }
                    uint32_t wa[16], wb[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        wa[e] = w[e];
                        wb[e] = w[e < 4 ? 16 + e : 0];  // 20 words
                    }
                    tmem_st16(tm + Gm::KEEP + 64 + 32 * hh, wa);
                    tmem_st16(tm + Gm::KEEP + 64 + 32 * hh + 16, wb);
                }
                if constexpr (K == 32) {
                    auto val = [&](int e) {
                        return e < 2 * N0 ? lane2(t0[e < 2 * N0 ? e / 2 : 0], e & 1)
                                          : lane2(t1[e < 2 * N0 ? 0 : (e - 2 * N0) / 2], e & 1);
                    };
#pragma unroll
                    for (int v = 0; v < 5; ++v)
                        kept[8 * (J * (J + 1) / 2 + J) + v] =
                            make_float4(val(4 * v), val(4 * v + 1), val(4 * v + 2), val(4 * v + 3));
                }
                if (J > 0) {  // less the earlier columns: four per step, loaded one step ahead
                    uint32_t a[2][16], b[2][16];
                    tmem_ld16(a[0], tcol(J, 0));
                    tmem_ld16(b[0], tcol(J, 0) + 32);
#pragma unroll 1
                    for (int kb = 0; kb < J; ++kb) {
                        float y[TB];
                        ln.floats(Gm::V, kb, y);
#pragma unroll
                        for (int s = 0; s < 2; ++s) {
                            tmem_wait_ld(a[s], b[s]);
                            if (s == 0) {
                                tmem_ld16(a[1], tcol(J, kb) + 16);
                                tmem_ld16(b[1], tcol(J, kb) + 48);
                            } else if (kb + 1 < J) {
                                tmem_ld16(a[0], tcol(J, kb + 1));
                                tmem_ld16(b[0], tcol(J, kb + 1) + 32);
                            }
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const uint32_t* o = (p0 == 0 ? a[s] : b[s]) + 4 * e;  // the owned rows
                                const u64 L0 = pk2u(o[0], o[1]), L1 = pk2u(o[2], o[3]);
#pragma unroll
                                for (int c = 0; c < N1; ++c) {
                                    const u64 m = dup2(__uint_as_float(
                                        half_of(c) ? b[s][4 * e + place_of(c)]
                                                   : a[s][4 * e + place_of(c)]));
                                    if (c < N0) t0[c] = fma2(L0, m, t0[c]);
                                    t1[c] = fma2(L1, m, t1[c]);
                                }
                                const u64 m = dup2(y[4 * s + e]);
                                nv[0] = fma2(L0, m, nv[0]);
                                nv[1] = fma2(L1, m, nv[1]);
                            }
                        }
                    }
                }
                // the tile to both threads: pair p, columns 2 i and 2 i + 1 in
                // vector 4 p + i
#pragma unroll
                for (int i = 0; i <= p0; ++i)
                    ln.vec(Gm::DG + 4 * p0 + i) =
                        make_float4(lo2(t0[2 * i]), hi2(t0[2 * i]), lo2(t0[2 * i + 1]), hi2(t0[2 * i + 1]));
#pragma unroll
                for (int i = 0; i <= p1; ++i)
                    ln.vec(Gm::DG + 4 * p1 + i) =
                        make_float4(lo2(t1[2 * i]), hi2(t1[2 * i]), lo2(t1[2 * i + 1]), hi2(t1[2 * i + 1]));
                ln.pair(Gm::XB + 2 * (J & 1), 0, p0) = make_float2(lo2(nv[0]), hi2(nv[0]));
                ln.pair(Gm::XB + 2 * (J & 1), 0, p1) = make_float2(lo2(nv[1]), hi2(nv[1]));
            };
            if (hh == 0)
                diag_part(std::integral_constant<int, 0>{});
            else
                diag_part(std::integral_constant<int, 1>{});
            pair_sync();
            {
                u64 t[TB][P], nvp[P];
#pragma unroll
                for (int q = 0; q < P; ++q)
#pragma unroll
                    for (int i = 0; i <= q; ++i) {
                        const float4 f = ln.vec(Gm::DG + 4 * q + i);
                        t[2 * i][q] = pk2(f.x, f.y);
                        t[2 * i + 1][q] = pk2(f.z, f.w);
                    }
                ln.pairs(Gm::XB + 2 * (J & 1), 0, nvp);
                float y[TB];
                factor_tile<TB>(t, nvp, Ld, ni, y);
                if (hh == 0) {
                    ln.put(Gm::V, J, y);
                    ln.put(Gm::DI, J, ni);
                } else {
                    uint32_t a[16], b[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        a[i] = __float_as_uint(Ld[i]);
                        b[i] = __float_as_uint(Ld[16 + i < Gm::TRI ? 16 + i : 0]);
                    }
                    tmem_st16(dcol(J), a);
                    tmem_st16(dcol(J) + 16, b);
                }
            }
#pragma unroll 1
            for (int I = J + 1; I < NB; ++I) {
                u64 t[2][8];
                assemble_off<K, kSph>(ln, vg, I, J, pr, ke, full, t);
                if constexpr (K == 16) {  // kept for the residual: a = -A' of the off-diagonal tile
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        uint32_t w[16];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                w[4 * e + 2 * u] = (uint32_t)__float2int_rn(lo2(t[u][4 * s + e]));
                                w[4 * e + 2 * u + 1] = (uint32_t)__float2int_rn(hi2(t[u][4 * s + e]));
                            }
                        tmem_st16(tm + Gm::KEEP + 32 * hh + 16 * s, w);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < TB; ++c)
                        kept[8 * (I * (I + 1) / 2 + J) + c] =
                            make_float4(lo2(t[0][c]), hi2(t[0][c]), lo2(t[1][c]), hi2(t[1][c]));
                }
                if (J > 0) {
                    uint32_t a[2][16], b[2][16], o[2][16];
                    tmem_ld16(a[0], tcol(J, 0));
                    tmem_ld16(b[0], tcol(J, 0) + 32);
                    tmem_ld16(o[0], tcol(I, 0) + 32 * hh);
#pragma unroll 1
                    for (int kb = 0; kb < J; ++kb) {
#pragma unroll
                        for (int s = 0; s < 2; ++s) {
                            tmem_wait_ld(a[s], b[s]);
                            tmem_use(o[s]);
                            if (s == 0) {
                                tmem_ld16(a[1], tcol(J, kb) + 16);
                                tmem_ld16(b[1], tcol(J, kb) + 48);
                                tmem_ld16(o[1], tcol(I, kb) + 32 * hh + 16);
                            } else if (kb + 1 < J) {
                                tmem_ld16(a[0], tcol(J, kb + 1));
                                tmem_ld16(b[0], tcol(J, kb + 1) + 32);
                                tmem_ld16(o[0], tcol(I, kb + 1) + 32 * hh);
                            }
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const u64 L0 = pk2u(o[s][4 * e], o[s][4 * e + 1]);
                                const u64 L1 = pk2u(o[s][4 * e + 2], o[s][4 * e + 3]);
#pragma unroll
                                for (int c = 0; c < 8; ++c) {
                                    const u64 m = dup2(__uint_as_float(
                                        half_of(c) ? b[s][4 * e + place_of(c)]
                                                   : a[s][4 * e + place_of(c)]));
                                    t[0][c] = fma2(L0, m, t[0][c]);
                                    t[1][c] = fma2(L1, m, t[1][c]);
                                }
                            }
                        }
                    }
                }
                // solve against the diagonal tile: X Ljj^T = A - ..., row by row
                int at = 0;
#pragma unroll
                for (int c = 0; c < TB; ++c) {
                    const u64 m = dup2(ni[c]);
                    t[0][c] = mul2(t[0][c], m);
                    t[1][c] = mul2(t[1][c], m);
#pragma unroll
                    for (int r = c + 1; r < TB; ++r) {
                        const u64 l = dup2(Ld[at++]);
                        t[0][r] = fma2(t[0][c], l, t[0][r]);
                        t[1][r] = fma2(t[1][c], l, t[1][r]);
                    }
                }
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    uint32_t a[16];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            a[4 * e + 2 * u] = __float_as_uint(lo2(t[u][4 * s + e]));
                            a[4 * e + 2 * u + 1] = __float_as_uint(hi2(t[u][4 * s + e]));
                        }
                    tmem_st16(tcol(I, J) + 32 * hh + 16 * s, a);
                }
            }
            pair_sync_tmem();
        }

        // ---- solve, one refinement step, solve again: the unknowns in registers
        // (the same in both threads); a tile row's sums are shared out and
        // exchanged through the two buffers XB in turn
        auto load_diag = [&](int J) {
            uint32_t a[16], b[16];
            tmem_ld16(a, dcol(J));
            tmem_ld16(b, dcol(J) + 16);
            ln.floats(Gm::DI, J, ni);
            tmem_wait_ld(a, b);
#pragma unroll
            for (int i = 0; i < Gm::TRI; ++i) Ld[i] = __uint_as_float(i < 16 ? a[i] : b[i - 16]);
        };
        float x[NB][TB];
        auto forward = [&]() {  // L y = v: thread hh brings -v of its row pairs in x's place
#pragma unroll
            for (int I = 0; I < NB; ++I) {
                u64 nv[2] = {pk2(x[I][0], x[I][1]), pk2(x[I][2], x[I][3])};
#pragma unroll
                for (int J = 0; J < I; ++J) {
                    uint32_t a[16], b[16];
                    tmem_ld16(a, tcol(I, J) + 32 * hh);
                    tmem_ld16(b, tcol(I, J) + 32 * hh + 16);
                    tmem_wait_ld(a, b);
#pragma unroll
                    for (int c = 0; c < TB; ++c) {
                        const uint32_t* w = c < 4 ? a + 4 * c : b + 4 * (c - 4);
                        const u64 m = dup2(x[J][c]);
                        nv[0] = fma2(pk2u(w[0], w[1]), m, nv[0]);
                        nv[1] = fma2(pk2u(w[2], w[3]), m, nv[1]);
                    }
                }
                load_diag(I);
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    ln.pair(Gm::XB + 2 * (I & 1), 0, pr[u]) = make_float2(lo2(nv[u]), hi2(nv[u]));
                pair_sync();
                ln.floats(Gm::XB + 2 * (I & 1), 0, x[I]);
                diag_forward<TB>(Ld, ni, x[I]);
            }
        };
        auto backward = [&]() {  // L^T x = y: thread hh brings y of columns 4 hh .. 4 hh + 3
#pragma unroll
            for (int J = NB - 1; J >= 0; --J) {
                u64 sum[4];  // owned columns; partial sums of the even and the odd rows
#pragma unroll
                for (int c = 0; c < 4; ++c) sum[c] = 0;
#pragma unroll
                for (int I = NB - 1; I > J; --I) {
                    uint32_t a[16], b[16];
                    tmem_ld16(a, tcol(I, J) + 16 * hh);
                    tmem_ld16(b, tcol(I, J) + 16 * hh + 32);
                    tmem_wait_ld(a, b);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        sum[c] = fma2(pk2u(a[4 * c], a[4 * c + 1]), pk2(x[I][0], x[I][1]), sum[c]);
                        sum[c] = fma2(pk2u(b[4 * c], b[4 * c + 1]), pk2(x[I][2], x[I][3]), sum[c]);
                        sum[c] = fma2(pk2u(b[4 * c + 2], b[4 * c + 3]), pk2(x[I][4], x[I][5]), sum[c]);
                        sum[c] = fma2(pk2u(a[4 * c + 2], a[4 * c + 3]), pk2(x[I][6], x[I][7]), sum[c]);
                    }
                }
                load_diag(J);
                const int buf = Gm::XB + 2 * ((NB - 1 - J) & 1);
                ln.vec(buf + hh) = make_float4(__fadd_rn(__fadd_rn(lo2(sum[0]), hi2(sum[0])), -x[J][0]),
                                               __fadd_rn(__fadd_rn(lo2(sum[1]), hi2(sum[1])), -x[J][1]),
                                               __fadd_rn(__fadd_rn(lo2(sum[2]), hi2(sum[2])), -x[J][2]),
                                               __fadd_rn(__fadd_rn(lo2(sum[3]), hi2(sum[3])), -x[J][3]));
                pair_sync();
                ln.floats(buf, 0, x[J]);
                diag_backward<TB>(Ld, ni, x[J]);
            }
        };
#pragma unroll
        for (int J = 0; J < NB; ++J) {
            const float4 y = ln.vec(Gm::V + 2 * J + hh);
            x[J][0] = y.x;
            x[J][1] = y.y;
            x[J][2] = y.z;
            x[J][3] = y.w;
        }
        backward();
        // The residual b - A' x' is exact: x' is x rounded to 24-bit fixed point
        // (representable in FP32), A' the 30-bit copy, and the sum of the
        // 2^54-bounded products is accumulated in 64-bit integers without rounding.
        float xmax = 0.0f;
#pragma unroll
        for (int I = 0; I < NB; ++I)
#pragma unroll
            for (int r = 0; r < TB; ++r) xmax = fmaxf(xmax, fabsf(x[I][r]));
        const int ex = xmax > 0.0f ? 24 - exp_above(xmax) : 0;
        const float sx = pow2f(ex), isx = pow2f(-ex);
        // (the solution of L y = b in V has been read by both threads: each passed
        // a barrier of the back substitution after it)
        if (hh == 0) {
#pragma unroll
            for (int I = 0; I < NB; ++I) {
                int xq[TB];
#pragma unroll
                for (int r = 0; r < TB; ++r) xq[r] = __float2int_rn(x[I][r] * sx);
                ln.put_ints(Gm::V, I, xq);
            }
        }
        pair_sync();
        const int acc0 = Gm::ACC + hh * 2 * Gm::Q;  // this thread's sums: pair p of row I at 4 I + p
        float4 nxt[8];  // the tile ahead
        int tile = 0;
        if constexpr (K == 32)
#pragma unroll
            for (int c = 0; c < 8; ++c) nxt[c] = kept[c];
#pragma unroll 1
        for (int I = 0; I < NB; ++I) {
            long long accr[4];
            int xi[TB], xr[4];
            ln.ints(Gm::V, I, xi);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float2 z = ln.pair(Gm::Z, I, pr[u]), g0 = ln.pair(Gm::G0, I, pr[u]),
                             xx = ln.pair(Gm::V, I, pr[u]);
                accr[2 * u] = float_to_ll(-minus_b(8 * I + 2 * pr[u], z.x, g0.x) * sx);
                accr[2 * u + 1] = float_to_ll(-minus_b(8 * I + 2 * pr[u] + 1, z.y, g0.y) * sx);
                xr[2 * u] = __float_as_int(xx.x);
                xr[2 * u + 1] = __float_as_int(xx.y);
            }
            // (the sums take + a x' with a = -A')
#pragma unroll 1
            for (int J = 0; J < I; ++J) {
                uint32_t qa[16], qb[16];
                float4 cur[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) cur[c] = nxt[c];
                if constexpr (K == 32) {
                    ++tile;
#pragma unroll
                    for (int c = 0; c < 8; ++c) nxt[c] = kept[8 * tile + c];
                }
                if constexpr (K == 16) {
                    tmem_ld16(qa, tm + Gm::KEEP + 32 * hh);
                    tmem_ld16(qb, tm + Gm::KEEP + 32 * hh + 16);
                    tmem_wait_ld(qa, qb);
                }
                int xj[TB];
                ln.ints(Gm::V, J, xj);
#pragma unroll
                for (int c2 = 0; c2 < 4; ++c2) {
                    longlong2 aj = ln.long2(acc0 + 4 * J + c2);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int c = 2 * c2 + e;
                        long long s = e ? aj.y : aj.x;
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            int a0, a1;
                            if constexpr (K == 16) {
                                a0 = (int)(c < 4 ? qa[4 * c + 2 * u] : qb[4 * (c - 4) + 2 * u]);
                                a1 = (int)(c < 4 ? qa[4 * c + 2 * u + 1] : qb[4 * (c - 4) + 2 * u + 1]);
                            } else {
                                a0 = __float2int_rn(u ? cur[c].z : cur[c].x);
                                a1 = __float2int_rn(u ? cur[c].w : cur[c].y);
                            }
                            accr[2 * u] += (long long)a0 * xj[c];
                            accr[2 * u + 1] += (long long)a1 * xj[c];
                            s += (long long)a0 * xr[2 * u];
                            s += (long long)a1 * xr[2 * u + 1];
                        }
                        if (e)
                            aj.y = s;
                        else
                            aj.x = s;
                    }
                    ln.long2(acc0 + 4 * J + c2) = aj;
                }
            }
            float4 cur[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) cur[c] = nxt[c];
            if constexpr (K == 32) {
                ++tile;
                if (I + 1 < NB)
#pragma unroll
                    for (int c = 0; c < 8; ++c) nxt[c] = kept[8 * tile + c];
            }
            auto diag_part = [&](auto which) {
                constexpr int p0 = decltype(which)::value, p1 = 3 - p0, N0 = 2 * p0 + 2, N1 = 2 * p1 + 2;
                long long acc[TB];
#pragma unroll
                for (int r = 0; r < TB; ++r) acc[r] = 0;
                acc[2 * p0] = accr[0];
                acc[2 * p0 + 1] = accr[1];
                acc[2 * p1] = accr[2];
                acc[2 * p1 + 1] = accr[3];
                // entries below the diagonal also stand for their mirror image
                auto add = [&](int r, int c, int a) {
                    acc[r] += (long long)a * xi[c];
                    if (r != c) acc[c] += (long long)a * xi[r];
                };
                auto add_tile = [&](auto at0, auto at1) {  // the entries of pair p0 and of pair p1
#pragma unroll
                    for (int c = 0; c < N0; ++c) {
                        if (c <= 2 * p0) add(2 * p0, c, at0(2 * c));
                        add(2 * p0 + 1, c, at0(2 * c + 1));
                    }
#pragma unroll
                    for (int c = 0; c < N1; ++c) {
                        if (c <= 2 * p1) add(2 * p1, c, at1(2 * c));
                        add(2 * p1 + 1, c, at1(2 * c + 1));
                    }
                };
                if (K == 16 && I == 0) {
                    uint32_t a[16], b[16];
                    tmem_ld16(a, tm + Gm::KEEP + 64 + 32 * hh);
                    tmem_ld16(b, tm + Gm::KEEP + 64 + 32 * hh + 16);
                    tmem_wait_ld(a, b);
                    add_tile([&](int e) { return (int)a[e]; },
                             [&](int e) { return (int)(2 * N0 + e < 16 ? a[2 * N0 + e] : b[2 * N0 + e - 16]); });
                } else if constexpr (K == 32) {
                    auto val = [&](int e) {
                        const float4 v = cur[e / 4];
                        return __float2int_rn(e % 4 == 0 ? v.x : e % 4 == 1 ? v.y : e % 4 == 2 ? v.z : v.w);
                    };
                    add_tile([&](int e) { return val(e); }, [&](int e) { return val(2 * N0 + e); });
                } else {
                    float xc[8], yc[8], zc[8];
                    ln.floats(Gm::X, I, xc);
                    ln.floats(Gm::Y, I, yc);
                    ln.floats(Gm::Z, I, zc);
                    u64 t0[N0], t1[N1];
                    assemble_diag<K, kSph, p0>(ln, vg, I, ke, sa, full, xc, yc, zc, t0);
                    assemble_diag<K, kSph, p1>(ln, vg, I, ke, sa, full, xc, yc, zc, t1);
                    add_tile([&](int e) { return __float2int_rn(lane2(t0[e / 2], e & 1)); },
                             [&](int e) { return __float2int_rn(lane2(t1[e / 2], e & 1)); });
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    ln.long2(acc0 + 4 * I + q) = make_longlong2(acc[2 * q], acc[2 * q + 1]);
            };
            if (hh == 0)
                diag_part(std::integral_constant<int, 0>{});
            else
                diag_part(std::integral_constant<int, 1>{});
        }
        pair_sync();
#pragma unroll
        for (int I = 0; I < NB; ++I)
#pragma unroll
            for (int u = 0; u < 2; ++u) {  // -sa (b - A' x') of the owned rows
                const longlong2 a = ln.long2(Gm::ACC + 4 * I + pr[u]);
                const longlong2 b = ln.long2(Gm::ACC + 2 * Gm::Q + 4 * I + pr[u]);
                x[I][2 * u] = -(ll_to_float(a.x + b.x) * isx);
                x[I][2 * u + 1] = -(ll_to_float(a.y + b.y) * isx);
            }
        forward();
        // y of the owned columns to the front, as backward() takes it
#pragma unroll
        for (int I = 0; I < NB; ++I)
#pragma unroll
            for (int c = 0; c < 4; ++c) x[I][c] = hh ? x[I][c + 4] : x[I][c];
        backward();

        // ---- weights and outputs: thread 0 the depth, thread 1 the variance. The
        // weight sum closes in FP64: x' sums exactly as integers (32 x 2^24), the
        // correction in FP32. Sums run in eight partials, combined pairwise.
        if (hh == 0) {
            float pz[TB];
#pragma unroll
            for (int r = 0; r < TB; ++r) pz[r] = 0.0f;
#pragma unroll
            for (int I = 0; I < NB; ++I) {
                float dz[TB];
                int xq[TB];
                ln.floats(Gm::DZ, I, dz);
                ln.ints(Gm::V, I, xq);
#pragma unroll
                for (int r = 0; r < TB; ++r)  // lambda (z_a - z_0)
                    pz[r] = fmaf(__fadd_rn(__fmul_rn((float)xq[r], isx), x[I][r]), dz[r], pz[r]);
            }
            if (live) depth[node] = ke == 0 ? __int_as_float(0x7fc00000) : z0 + idw_tree8(pz);  // no valid sounding: NaN
        } else if (var) {
            int sq = 0;
            float ps[TB], pv[TB];
#pragma unroll
            for (int r = 0; r < TB; ++r) ps[r] = pv[r] = 0.0f;
#pragma unroll
            for (int I = 0; I < NB; ++I) {
                float g0[TB], z[TB];
                int xq[TB];
                ln.floats(Gm::G0, I, g0);
                ln.floats(Gm::Z, I, z);
                ln.ints(Gm::V, I, xq);
#pragma unroll
                for (int r = 0; r < TB; ++r) {
                    const float lam = __fadd_rn(__fmul_rn((float)xq[r], isx), x[I][r]);
                    sq += xq[r];
                    ps[r] = __fadd_rn(ps[r], x[I][r]);
                    pv[r] = fmaf(lam, __fadd_rn(g0[r], z[r] * isa), pv[r]);  // gamma_0a - Gamma_a0
                }
            }
            const float lam0 = (float)(1.0 - ((double)sq * (double)isx + (double)idw_tree8(ps)));
            if (live)
                var[node] = ke == 0 ? __int_as_float(0x7fc00000) : fmaf(lam0, g00, g00 + idw_tree8(pv));
        }
        pair_sync_tmem();  // the next batch overwrites the records and the factor
    }
    }
}

}  // namespace bg
