// Exact k-nearest-neighbour search of 32 nearby nodes by one warp.
//
// A warp takes a patch of 8 x 4 grid nodes, one node per lane,
// and walks a strip of patches along x. Neighbouring nodes share almost all
// their candidates, so the candidates of the whole patch are staged once and
// every lane tests each of them, without divergence:
//   1. a radius per lane: from the density around the patch (summed-area
//      table), later from the lane's neighbour distances in the previous patch;
//      where that misses by far (soundings to one side, clusters), from the exact
//      neighbours of a node in the middle, found by the whole warp (knn_query.cuh);
//   2. the records of every cell run that can hold a point within the largest
//      radius of the patch go to shared memory (coalesced loads);
//   3. each lane computes its squared distance to each staged record (a
//      broadcast read, 32-bit integers) and appends those within its radius to
//      its column of a buffer, as 32-bit keys: distance above, place in the
//      staged list below (9 bits);
//   4. the search is exact when at least K were appended and none was lost: a
//      lane with fewer than K or with more than the buffer holds moves its
//      radius and the patch is scanned again;
//   5. the K smallest keys come from compare-exchange networks in registers:
//      blocks of K sorted (odd-even merge), each merged into the best so far.
// The keys order by distance and then by staged place, so equal distances are
// put in (distance, upload index) order afterwards, from the exact values; so
// are distances that a key holds only in part (large radii drop low bits).
//
// What bounds it: latency at 16 (K <= 16) or 12 (K = 32) resident warps per
// SM, half of the issue slots used (18 warps of 96 registers instead of 16 of 128 spill:
// whole pass of the swath below 1.40 ms, 1.28 so); a per-thread heap was bound by divergence.
// IDW k = 16 on a two-line swath (4,000 x 1,692 nodes, a 154 m gap): a heap per
// thread 277 warp instructions per node with 16 of 32 lanes active, 2.04 ms;
// this search 102 with 30, 1.17 ms. A candidate costs a warp 7 instructions for
// its 32 nodes (114 per patch there, 1.15 scans), the networks about 550 a
// patch. The straight path is kept short (rare courses in functions of their
// own): with everything inlined the instruction cache missed on three of four
// issues and the same search took 3.3 ms.
// Uneven soundings, us by threads / with the density's radius alone / so: 256 x 256
// nodes k = 8, half of the box empty 106 / 137 / 95, the other half denser 153 / 191 /
// 123, eight of the former in a batch 418 / 730 / 371; 500 x 500 over clusters 224 / 286 /
// 199; single-beam lines 500 m apart, 400 x 350 nodes k = 16 467 / 690 / 385, 2,000 x
// 1,900 over denser ones 11,032 / 31,418 / 12,342.
// Patches the staged list cannot hold (many soundings per node), nodes far
// outside the data and the like are left to the caller's per-thread search.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "knn.cuh"
#include "knn_query.cuh"

namespace bg {

// Staged records per patch, buffer rows per lane (with the slack of one
// unrolled step), and the radius the first patch of a strip starts with, as a
// multiple of the area that holds K soundings at the local density (about three
// standard deviations of a random count above K).
template <int K>
struct KnnWarp {
    static constexpr int kStep = 8;  // candidates per unrolled step
    static constexpr int CAP = K == 32 ? 320 : 256;
    static constexpr int ROWS = K == 32 ? 80 : K == 16 ? 48 : 40;
    static constexpr int B = ROWS - kStep;
    static constexpr float kArea = K == 32 ? 1.6f : K == 16 ? 1.9f : K == 8 ? 2.2f : 3.0f;
    static constexpr int kBlocksPerSM = K == 32 ? 6 : 8;  // of two warps: by shared memory
    struct Smem {
        uint32_t buf[ROWS * 32];  // column per lane (the per-thread heap, 8 K bytes, fits too)
        int4 st[CAP];             // {x, y relative to the patch, x^2 + y^2, place}
        int pos[CAP];             // record
    };
    // (the last block of K rows may end past the buffer: in the list, unused)
    static_assert(ROWS * 4 >= 8 * K && CAP % kStep == 0 && CAP >= 8 * K, "buffer rows");
};
constexpr int kPlaceBits = 9;
constexpr uint32_t kNoKey = 0xffffffffu;

__device__ __forceinline__ void cswap(uint32_t& a, uint32_t& b) {
    const uint32_t lo = min(a, b), hi = max(a, b);
    a = lo;
    b = hi;
}
// odd-even merge sort (Batcher) of v[LO .. LO + N), ascending
template <int LO, int N, int R, int K>
__device__ __forceinline__ void net_merge(uint32_t (&v)[K]) {
    constexpr int M = 2 * R;
    if constexpr (M < N) {
        net_merge<LO, N, M>(v);
        net_merge<LO + R, N, M>(v);
#pragma unroll
        for (int i = LO + R; i + R < LO + N; i += M) cswap(v[i], v[i + R]);
    } else {
        cswap(v[LO], v[LO + R]);
    }
}
template <int LO, int N, int K>
__device__ __forceinline__ void net_sort(uint32_t (&v)[K]) {
    if constexpr (N > 1) {
        net_sort<LO, N / 2>(v);
        net_sort<LO + N / 2, N / 2>(v);
        net_merge<LO, N, 1>(v);
    }
}
// ascending order of a bitonic v[LO .. LO + N)
template <int LO, int N, int K>
__device__ __forceinline__ void net_bitonic(uint32_t (&v)[K]) {
    if constexpr (N > 1) {
#pragma unroll
        for (int i = LO; i < LO + N / 2; ++i) cswap(v[i], v[i + N / 2]);
        net_bitonic<LO, N / 2>(v);
        net_bitonic<LO + N / 2, N / 2>(v);
    }
}

// Append `key` at shared address `a` (the lane's buffer column) when d <= lim:
// predicated, without a branch.
__device__ __forceinline__ void append_if(int d, int lim, uint32_t key, uint32_t& a) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.le.s32 p, %1, %2;\n\t"
        "@p st.shared.b32 [%0], %3;\n\t"
        "@p add.u32 %0, %0, 128;\n\t}"
        : "+r"(a)
        : "r"(d), "r"(lim), "r"(key)
        : "memory");
}
__device__ __forceinline__ void append_if(uint32_t d, uint32_t lim, uint32_t key, uint32_t& a) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.le.u32 p, %1, %2;\n\t"
        "@p st.shared.b32 [%0], %3;\n\t"
        "@p add.u32 %0, %0, 128;\n\t}"
        : "+r"(a)
        : "r"(d), "r"(lim), "r"(key)
        : "memory");
}

// What a lane carries from one patch of its strip to the next.
struct KnnChain {
    float d1 = 0.0f, dk = -1.0f;  // distances (cm) to its nearest (a lower bound) and K-th; dk < 0: none
    float beta = 1.2f;            // warp: (r - d1) / (dk - d1) tried next
};

constexpr uint32_t kPlaceMask = (1u << kPlaceBits) - 1;

// Soundings density around hash cell (cx, cy): the radius (cm) whose disc holds
// about `want` soundings, from the smallest of 32 squares (one per lane) that
// holds 4 want; < 0 when none does.
__device__ __forceinline__ float density_radius(const HashView& h, int cx, int cy, float want) {
    const int lane = threadIdx.x & 31;
    const int need = (int)fminf(4.0f * want, 0.5f * (float)h.n_valid);
    int w = h.r0 + lane;
#pragma unroll 1
    for (int round = 0; round < 2; ++round) {
        const int xa = max(cx - w, 0), xb = min(cx + w, h.ncx - 1);
        const int ya = max(cy - w, 0), yb = min(cy + w, h.ncy - 1);
        const int c = sat_count(h, xa, ya, xb, yb);
        const unsigned ok = __ballot_sync(kFull, c >= need);
        if (ok) {
            const float cells = (float)(xb - xa + 1) * (float)(yb - ya + 1);
            const float a = want * cells * (float)h.cs * (float)h.cs / (3.14159265f * (float)max(c, 1));
            return sqrtf(__shfl_sync(kFull, a, __ffs(ok) - 1));
        }
        w = h.r0 + 32 + 32 * lane;
    }
    return -1.0f;
}

// The first radius of each lane for a patch `step` cm further along the strip
// (from the distances it carries), and a lower bound `base` of its squared
// distances; without them, from the density around the patch.
template <int K>
__device__ __forceinline__ float knn_first_radius(const HashView& h, const KnnChain& ch, bool on, int qx,
                                                  int qy, float step, uint32_t& base) {
    base = 0;
    const bool have = on && ch.dk >= 0.0f;
    if (__all_sync(kFull, have || !on)) {
        // the patch's mean where the lanes are alike and surrounded by soundings
        // (less noise), else the lane's own
        const float mx = __uint_as_float(__reduce_max_sync(kFull, have ? __float_as_uint(ch.dk) : 0u));
        const float mn = __uint_as_float(__reduce_min_sync(kFull, have ? __float_as_uint(ch.dk) : 0x7f7fffffu));
        const float m1 = __uint_as_float(__reduce_max_sync(kFull, have ? __float_as_uint(ch.d1) : 0u));
        if (mx < 1.6f * mn && m1 < 0.7f * mn) {
            float s = have ? ch.dk : 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
            return s / (float)max(1, __popc(__ballot_sync(kFull, have))) * ch.beta + 1.0f;
        }
        const float f = fmaxf(0.0f, ch.d1 * 0.99999f - step - 1.0f);
        base = have ? (uint32_t)(f * f) : 0u;
        return ch.d1 + (ch.dk - ch.d1) * fmaxf(1.3f, ch.beta) + 1.0f;
    }
    const unsigned m = __ballot_sync(kFull, on);
    const int src = m == kFull ? 12 : 31 - __clz(m | 1);  // a node of the patch; its middle for a whole one
    const int cx = clamp_cell(h, (int64_t)__shfl_sync(kFull, qx, src) - h.hx0, h.ncx);
    const int cy = clamp_cell(h, (int64_t)__shfl_sync(kFull, qy, src) - h.hy0, h.ncy);
    return density_radius(h, cx, cy, KnnWarp<K>::kArea * K);
}

__device__ __forceinline__ int4 staged(int x, int y, int place) {
    return make_int4(x, y, (int)((uint32_t)(x * x) + (uint32_t)(y * y)), place);
}

// Bounds of the 32-bit squared distances, in cm: radius, patch and hash cell. The
// far scan takes only records within a lane's radius along each axis (d < 2^32);
// the near scan, in signed sums of the staged squares, needs every staged record
// within kNearMax of every node along each axis.
constexpr int kRadiusMax = 46000, kPatchMax = 10000, kCellMax = 30000, kNearMax = 26000;

// Stage every record within the radii of the patch (r of the lanes with `on`,
// at (ux, uy) relative to the corner (ox, oy)); returns their number, or -1 when
// there are more than the list holds.
template <int K>
__device__ __forceinline__ int knn_stage(const HashView& h, typename KnnWarp<K>::Smem& sm, bool on, int ux,
                                         int uy, int ox, int oy, float r) {
    using W = KnnWarp<K>;
    const int lane = threadIdx.x & 31;
    // largest radius of each 8-lane group (a row of a grid patch), and its y range
    const int ri = on ? __float2int_ru(r) : 0;
    int rg = ri, yg = on ? uy : INT_MAX, yh = on ? uy : INT_MIN;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        rg = max(rg, __shfl_xor_sync(kFull, rg, o));
        yg = min(yg, __shfl_xor_sync(kFull, yg, o));
        yh = max(yh, __shfl_xor_sync(kFull, yh, o));
    }
    // Circles of the largest radius about [xmin, xmax] hold every lane's: of circles that
    // reach as far along x, the largest falls back least above and below. (Where the
    // soundings lie to one side the radii differ by as much as the nodes' places, and
    // circles about those would reach in that much deeper.)
    const int xmin = __reduce_min_sync(kFull, on ? ux - ri + rg : INT_MAX);
    const int xmax = __reduce_max_sync(kFull, on ? ux + ri - rg : INT_MIN);
    const int ylo = __reduce_min_sync(kFull, yg <= yh ? yg - rg : INT_MAX);
    const int yhi = __reduce_max_sync(kFull, yg <= yh ? yh + rg : INT_MIN);
    // the corner relative to the hash (both lie in (-2^30, 2^30) cm)
    const int64_t cx = (int64_t)ox - h.hx0, cy = (int64_t)oy - h.hy0;
    const int ra = clamp_cell(h, cy + ylo, h.ncy), rb = clamp_cell(h, cy + yhi, h.ncy);
    const int wlast = h.ncx * h.cs - 1;  // last column of the hash, cm
    int T = 0;
    __syncwarp();  // the previous patch's readers are done with the list
#pragma unroll 1
    for (int row0 = ra; row0 <= rb; row0 += 32) {
        const int row = row0 + lane;
        const int64_t yr = (int64_t)row * h.cs - cy;  // the row's lower edge, relative to the patch
        const int yl = (int)max((int64_t)-(1 << 30), min((int64_t)(1 << 30), yr)), yu = yl + h.cs - 1;
        int dx2 = -1;
#pragma unroll
        for (int q = 0; q < 32; q += 8) {
            const int ga = __shfl_sync(kFull, yg, q), gb = __shfl_sync(kFull, yh, q), gr = __shfl_sync(kFull, rg, q);
            const int dy = max(0, max(yl - gb, ga - yu));
            if (ga <= gb && dy <= gr) dx2 = max(dx2, gr * gr - dy * dy);
        }
        int s = 0, len = 0;
        if (row <= rb && dx2 >= 0) {
            const int dxm = __float2int_ru(sqrtf((float)dx2) * 1.000002f) + 1;
            const int64_t xa = max(cx + (xmin - dxm), (int64_t)0), xb = min(cx + (xmax + dxm), (int64_t)wlast);
            if (xa <= xb) {
                const int* cs = h.cell_start + row * h.ncx;
                s = __ldg(cs + cell_of(h, xa));
                len = __ldg(cs + cell_of(h, xb) + 1) - s;
            }
        }
        int inc = len;  // records of the rows up to this lane's
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += v;
        }
        const int total = __shfl_sync(kFull, inc, 31);
        if (total > W::CAP - T) return -1;
        const int sb = s - (inc - len);
        // two records per lane in flight
#pragma unroll 1
        for (int i0 = lane; i0 - lane < total; i0 += 64) {
            int l0 = 0, l1 = 0;  // the rows that hold records i0 and i0 + 32 of this group
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                if (__shfl_sync(kFull, inc, l0 + o - 1) <= i0) l0 += o;
                if (__shfl_sync(kFull, inc, l1 + o - 1) <= i0 + 32) l1 += o;
            }
            const int p0 = __shfl_sync(kFull, sb, l0 & 31) + i0, p1 = __shfl_sync(kFull, sb, l1 & 31) + i0 + 32;
            int4 v0, v1;
            if (i0 < total) v0 = __ldg(h.rec + p0);
            if (i0 + 32 < total) v1 = __ldg(h.rec + p1);
            const int t = T + i0;
            if (i0 < total) {
                sm.st[t] = staged(v0.x - ox, v0.y - oy, t);
                sm.pos[t] = p0;
            }
            if (i0 + 32 < total) {
                sm.st[t + 32] = staged(v1.x - ox, v1.y - oy, t + 32);
                sm.pos[t + 32] = p1;
            }
        }
        T += total;
    }
    // to a whole step, beyond any radius
    if (lane < W::kStep && T + lane < W::CAP) sm.st[T + lane] = make_int4(60000, 0, 0x7fff0000, 0);
    __syncwarp();
    return T;
}

// (distance, upload index) order of two keys, from the exact values (after
// knn_stage_indices)
template <class Smem>
__device__ __forceinline__ bool key_less(const Smem& sm, int ux, int uy, uint32_t a, uint32_t b) {
    const int4 ca = sm.st[a & kPlaceMask], cb = sm.st[b & kPlaceMask];
    const int ax = ca.x - ux, ay = ca.y - uy, bx = cb.x - ux, by = cb.y - uy;
    const int da = ax * ax + ay * ay, db = bx * bx + by * by;
    return da != db ? da < db : ca.z < cb.z;
}
// The upload indices of the staged records in place of their squares; all lanes.
template <class Smem>
__device__ __forceinline__ void knn_stage_indices(Smem& sm, const int4* rec, int T) {
#pragma unroll 2
    for (int i = threadIdx.x & 31; i < T; i += 32) sm.st[i].z = __ldg(&rec[sm.pos[i]].w);
    __syncwarp();
}

// An appended word as the key it sorts by. The near scan appends 512 (d - u^2) +
// place, modulo 2^32, and the bias 512 (u^2 - base) makes it 512 (d - base) +
// place; the far scan appends the key itself (bias 0).
__device__ __forceinline__ uint32_t sort_key(uint32_t v, uint32_t bias) { return v + bias; }

// Of a lane's cnt appended keys those at the distance (as far as keys hold it) of the
// K-th, dk: the m nearest in exact order to the rows K - m .. K - 1 of its buffer
// column. Out of the way of the search's straight path. On a lattice every node comes
// here (511 x 511 nodes k = 32 over one of 2 m: 123 us; 469 with all keys sorted anew
// and indices from global memory, 201 by threads).
template <int K, class Smem>
__device__ __noinline__ void knn_last_group(Smem& sm, int ux, int uy, int cnt, int m, uint32_t dk, uint32_t bias) {
    uint32_t* buf = sm.buf + (threadIdx.x & 31);
    int n = 0;
    for (int i = 0; i < cnt; ++i) {
        const uint32_t v = sort_key(buf[i * 32], bias);
        if ((v ^ dk) <= kPlaceMask) buf[n++ * 32] = v;
    }
    // (K - m + n <= cnt: no row past the appended ones)
    for (int i = n - 1; i >= 0; --i) buf[(K - m + i) * 32] = buf[i * 32];
    buf += (K - m) * 32;
    for (int i = 1; i < n; ++i) {
        const uint32_t v = buf[i * 32];
        if (i >= m && !key_less(sm, ux, uy, v, buf[(m - 1) * 32])) continue;
        int j = min(i, m - 1);
        for (; j > 0 && key_less(sm, ux, uy, v, buf[(j - 1) * 32]); --j) buf[j * 32] = buf[(j - 1) * 32];
        buf[j * 32] = v;
    }
}

// For each lane's node a radius (cm) that holds K soundings, ub, and one that holds fewer,
// lo, from the exact K nearest of lane src's node: ub reaches all of those, lo is short
// of the K-th by the way between the nodes. r: the radius that failed. ub < 0: none.
struct KnnBracket {
    float lo, ub;
};
template <int K>
__device__ __noinline__ KnnBracket knn_centre(const HashView& h, int qx, int qy, float r, int src, uint64_t* buf) {
    const int sx = __shfl_sync(kFull, qx, src), sy = __shfl_sync(kFull, qy, src);
    uint64_t key = 0;
    // (off the data: its nodes share little)
    if (query_outside((int64_t)sx - h.hx0, (int64_t)sy - h.hy0, h.cs, h.ncx, h.ncy) > 4.0f * r) return KnnBracket{0.0f, -1.0f};
    if (knn_query<32>(h, true, sx, sy, K, buf, key) != K) return KnnBracket{0.0f, -1.0f};
    int4 p = make_int4(0, 0, 0, 0);
    if ((threadIdx.x & 31) < K) p = __ldg(h.orig + (key & ((1ull << h.idx_bits) - 1)));
    float most = 0.0f;
#pragma unroll 4
    for (int i = 0; i < K; ++i) {
        const float dx = (float)(__shfl_sync(kFull, p.x, i) - qx), dy = (float)(__shfl_sync(kFull, p.y, i) - qy);
        most = fmaxf(most, fmaf(dx, dx, dy * dy));
    }
    const float wx = (float)(qx - sx), wy = (float)(qy - sy);
    const float d = sqrtf((float)(__shfl_sync(kFull, key, K - 1) >> h.idx_bits));
    return KnnBracket{fmaxf(0.0f, 0.999999f * (d - sqrtf(wx * wx + wy * wy)) - 1.0f), 1.000001f * sqrtf(most) + 1.0f};
}

// The K nearest of each lane's node (qx, qy), for lanes with `on`; (ox, oy)
// is the patch's corner (the staged coordinates are relative to it; no node
// lies before it). r: the lane's first radius (cm; < 0: none), base: a lower
// bound of its squared distances; lo: a radius known to hold fewer than K. probe: what
// the caller can better with another radius, 0 nothing, 1 more records than the list
// holds, 2 also a radius far too small. No lane is served then and probe stays as it
// was; else it becomes 0. Returns the lanes that were served: the low
// kPlaceBits of the first K rows of their buffer columns index the staged list
// in ascending (distance, upload index) order.
template <int K>
__device__ __forceinline__ unsigned knn_patch(const HashView& h, typename KnnWarp<K>::Smem& sm, bool on,
                                              int qx, int qy, int ox, int oy, float r, uint32_t base,
                                              float lo, int& probe, KnnChain& ch) {
    using W = KnnWarp<K>;
    constexpr int B = W::B, S = W::kStep;
    const int lane = threadIdx.x & 31;
    const int ux = qx - ox, uy = qy - oy;
    constexpr float kMaxR = (float)kRadiusMax;
    on = on && r >= 0.0f && r < kMaxR && (unsigned)ux < (unsigned)kPatchMax && (unsigned)uy < (unsigned)kPatchMax;
    if (!__any_sync(kFull, on)) return 0;  // (a probe too: the caller finds another radius)
    uint32_t* buf = sm.buf + lane;
    const uint32_t buf0 = (uint32_t)__cvta_generic_to_shared(buf);
    float hi = 1e30f;  // a radius known to hold too many
    const float d0 = sqrtf((float)base);
    const int u2 = on ? ux * ux + uy * uy : 0;
    const uint32_t mx2 = on ? -2 * ux : 0, my2 = on ? -2 * uy : 0;  // (sums wrap, results fit)
    uint32_t bias = 0;
    int T = 0, cnt = 0, sh = 0;
    bool stage = true, grew = false, shrunk = false, full = false;
#pragma unroll 1
    for (int it = 0;; ++it) {
        if (stage) T = knn_stage<K>(h, sm, on, ux, uy, ox, oy, r);
        bool few = false, over = false;
        if (T >= 0) {
            // d = |c|^2 - 2 c u + |u|^2
            const int tau = (int)(r * r);
            // low bits of a distance that the key does not hold (none up to 28.9 m)
            sh = max(0, kPlaceBits - __clz(__reduce_max_sync(kFull, on ? (uint32_t)tau - base : 0u)));
            uint32_t at = buf0;
            auto scan = [&](auto append) {
#pragma unroll 1
                for (int i = 0; i < T; i += S) {  // the buffer has S rows of slack
#pragma unroll
                    for (int u = 0; u < S; ++u) {
                        const int4 c = sm.st[i + u];
                        append((uint32_t)c.x * mx2 + ((uint32_t)c.y * my2 + (uint32_t)c.z), (uint32_t)c.w, c);
                    }
                    over |= at > buf0 + B * 128;
                    at = min(at, buf0 + B * 128);
                }
            };
            // (near: every staged record within kNearMax)
            if (__all_sync(kFull, !on || r + (float)(kPatchMax + h.cs) < (float)kNearMax) && sh == 0) {
                // compared less |u|^2, in signed arithmetic
                const int lim = on ? tau - u2 : INT_MIN;
                bias = ((uint32_t)u2 - base) << kPlaceBits;
                scan([&](uint32_t d, uint32_t place, const int4&) {
                    append_if((int)d, lim, d * (1u << kPlaceBits) + place, at);
                });
            } else {
                const uint32_t lim = on ? (uint32_t)tau - base : 0u;
                const int R = on ? __float2int_ru(r) : 0;
                bias = 0;
                scan([&](uint32_t, uint32_t place, const int4& c) {
                    const int dx = c.x - ux, dy = c.y - uy;
                    const bool box = (unsigned)(dx + R) <= 2u * R && (unsigned)(dy + R) <= 2u * R;
                    const uint32_t e = (uint32_t)dx * dx + (uint32_t)dy * dy - base;
                    append_if(box ? e : kNoKey, lim, (e >> sh) * (1u << kPlaceBits) + place, at);
                });
            }
            cnt = (int)(at - buf0) / 128;
            over = on && over;
            few = on && !over && cnt < K;
        } else {  // more than the list holds: smaller radii for lanes that have missed below
            over = on && lo > 0.0f;
            if (full || probe != 0 || !__any_sync(kFull, over)) return 0;
            full = true;
        }
        if (probe == 2 && __any_sync(kFull, few && (it == 0 ? cnt == 0 : 2 * cnt <= K))) return 0;
        if (!__any_sync(kFull, few || over)) break;
        if (it >= 7) {
            if (T < 0) return 0;
            if (few || over) on = false;
            break;
        }
        // move the radii of the lanes that missed; the others scan again as they were
        stage = T < 0 || __any_sync(kFull, few);
        grew |= __any_sync(kFull, few);
        shrunk |= __any_sync(kFull, over);
        if (few) {
            lo = r;
            r = hi < 1e29f ? 0.5f * (lo + hi) : d0 + (r - d0) * (2 * cnt > K ? 1.25f : 1.6f) + 1.0f;
            if (r >= kMaxR) on = false;
        } else if (over) {
            hi = r;
            r = lo > 0.0f ? 0.5f * (lo + hi) : d0 + (hi - d0) * 0.85f;
        }
    }
    probe = 0;
    const unsigned served = __ballot_sync(kFull, on);
    if (served == 0) return 0;

    // the K smallest keys, ascending; drop: the smallest key left out
    uint32_t key[K], v[K], drop = kNoKey;
    const int blocks = (__reduce_max_sync(kFull, on ? cnt : 0) + K - 1) / K;
#pragma unroll 1
    for (int b = 0; b < blocks; ++b) {
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const uint32_t w = buf[(b * K + i) * 32];
            v[i] = b * K + i < cnt ? sort_key(w, bias) : kNoKey;
        }
        net_sort<0, K>(v);
        if (b == 0) {
#pragma unroll
            for (int i = 0; i < K; ++i) key[i] = v[i];
        } else {
#pragma unroll
            for (int i = 0; i < K; ++i) {
                drop = min(drop, max(key[i], v[K - 1 - i]));
                key[i] = min(key[i], v[K - 1 - i]);
            }
            net_bitonic<0, K>(key);
        }
    }
    // for the next patch: this lane's nearest (rounded down) and K-th distance, and
    // a wider or narrower first radius
    if (on) {
        ch.d1 = sqrtf((float)(((key[0] >> kPlaceBits) << sh) + base));
        ch.dk = sqrtf((float)(((key[K - 1] >> kPlaceBits) << sh) + base));
    } else {
        ch.dk = -1.0f;
    }
    const int least = __reduce_min_sync(kFull, on ? cnt : INT_MAX);
    if (grew)
        ch.beta = fminf(1.7f, ch.beta * 1.06f);
    else if (shrunk || least > K + K / 8 + 1)
        ch.beta = fmaxf(1.04f, ch.beta * (shrunk ? 0.96f : 0.99f));

    // equal distances (as far as the keys hold them): into (distance, index)
    // order, in place; where a key left out shares the K-th distance, from all that do
    const bool last = on && (key[K - 1] ^ drop) <= kPlaceMask;
    bool pair = false;
#pragma unroll
    for (int i = 0; i + 1 < K; ++i) pair |= (key[i] ^ key[i + 1]) <= kPlaceMask;
    int put = K;  // keys that are in place but for pairs
    if (__any_sync(kFull, last || (on && pair))) {
        knn_stage_indices(sm, h.rec, T);
        if (last) {
            put = 0;
#pragma unroll
            for (int i = 0; i < K; ++i) put += (key[i] ^ key[K - 1]) > kPlaceMask;
            knn_last_group<K>(sm, ux, uy, cnt, K - put, key[K - 1], bias);
        }
    }
#pragma unroll
    for (int i = 0; i < K; ++i)
        if (i < put) buf[i * 32] = key[i];
    if (on && pair) {
#pragma unroll 1
        for (int i = 1; i < put; ++i) {
            const uint32_t v = buf[i * 32];
            int j = i;
#pragma unroll 1
            for (; j > 0; --j) {
                const uint32_t u = buf[(j - 1) * 32];
                if ((u ^ v) > kPlaceMask || !key_less(sm, ux, uy, v, u)) break;
                buf[j * 32] = u;
            }
            if (j < i) buf[j * 32] = v;
        }
    }
    __syncwarp();
    return served;
}

// The per-thread search of one node for a lane that knn_patch did not serve:
// its packed keys sorted ascending in hp (stride 32); returns their number, or
// -1 when the bound does not fit a packed key. ub: a radius known to hold K soundings,
// < 0: none. Lanes run it on their own. Out of the way of the patch search's code.
template <int K>
__device__ __noinline__ int knn_lane(const HashView& h, int qx, int qy, uint64_t* hp, float ub) {
    if (ub >= 0.0f && ub < 2e9f) {
        const Bound t{(int64_t)(1.000001f * ub * ub) + 1, clamp_cell(h, (int64_t)qy - h.hy0, h.ncy), 0, 0};
        if (packed_fits(h, t.tau0)) {
            const int cnt = knn_scan_heap_rt<32, true>(h, qx, qy, t, hp, K);
            if (cnt == K) return cnt;
        }
    }
    const Bound b = knn_bound_rt(h, qx, qy, K);
    if (!packed_fits(h, b.tau0)) return -1;
    Bound bt = b;
    if (b.count > 0)  // as in knn_strip: 1.5 times the area at the square's density first
        bt.tau0 = min(b.tau0, (int64_t)fminf(1.5f * (float)K * (float)b.area / (3.14159265f * (float)b.count), 9e18f));
    for (;;) {
        const int cnt = knn_scan_heap_rt<32, true>(h, qx, qy, bt, hp, K);
        if (cnt == K || bt.tau0 == b.tau0) return cnt;
        bt.tau0 = b.tau0;
    }
}

// What a lane's own search (a node that knn_patch did not serve) found.
struct KnnFar {
    int cnt;       // neighbours; -1: left to the wide pass
    float d1, dk;  // distances to the nearest and the K-th (cnt == K)
};
template <int K>
__device__ __forceinline__ KnnFar knn_far(const HashView& h, const uint64_t* hp, int cnt) {
    return KnnFar{cnt, cnt > 0 ? sqrtf((float)(hp[0] >> h.idx_bits)) : 0.0f,
                  cnt == K ? sqrtf((float)(hp[(K - 1) * 32] >> h.idx_bits)) : 0.0f};
}

// Patches p0 .. p1 - 1 of the patch row whose first grid row is jb (rows below
// j1), one after another by one warp. served(i, j, ux, uy) runs for the nodes
// that the patch search served (knn_patch: the lane's buffer column and the
// staged list hold the neighbours), lone(i, j, qx, qy, heap, ub) for the others:
// it searches by itself (knn_lane) and returns a KnnFar. flag is set when a node
// is left to the wide pass (NULL: packed_always holds).
template <int K, class Served, class Lone>
__device__ __forceinline__ void knn_patch_row(const HashView& h, const GridView& g, typename KnnWarp<K>::Smem& sm,
                                              int jb, int j1, int p0, int p1, int* flag, Served served, Lone lone) {
    const int lane = threadIdx.x & 31;
    const int j = jb + (lane >> 3), qy = g.y0 + j * g.cell + g.cell / 2;
    KnnChain ch;
#pragma unroll 1
    for (int p = p0; p < p1 && p * 8 < g.nx; ++p) {
        const int i = p * 8 + (lane & 7), qx = g.x0 + i * g.cell + g.cell / 2;
        const bool on = i < g.nx && j < j1;
        const int ox = g.x0 + p * 8 * g.cell + g.cell / 2, oy = g.y0 + jb * g.cell + g.cell / 2;
        uint32_t base;
        const float step = 8.0f * (float)g.cell;
        int probe = __all_sync(kFull, !on || ch.dk >= 0.0f) ? 1 : 2;
        float ub = ch.dk >= 0.0f ? 1.000001f * (ch.dk + step) + 2.0f : -1.0f, lo = 0.0f;
        float r = knn_first_radius<K>(h, ch, on, qx, qy, step, base);
        unsigned m;
        for (;;) {
            m = knn_patch<K>(h, sm, on, qx, qy, ox, oy, r, base, lo, probe, ch);
            if (probe == 0) break;
            // the exact neighbours of a node in the middle bound every lane's
            probe = 0;
            __syncwarp();
            const unsigned all = __ballot_sync(kFull, on);
            const int src = all == kFull ? 12 : 31 - __clz(all);
            const KnnBracket b = knn_centre<K>(h, qx, qy, fmaxf(0.0f, __shfl_sync(kFull, r, src)), src,
                                               reinterpret_cast<uint64_t*>(sm.buf));
            lo = b.lo;
            r = ub = b.ub;
            base = 0;
        }
        if (m >> lane & 1) served(i, j, qx - ox, qy - oy);
        if (m != kFull) {
            __syncwarp();
            if (on && !(m >> lane & 1)) {
                ch.dk = -1.0f;
                const KnnFar f = lone(i, j, qx, qy, reinterpret_cast<uint64_t*>(sm.buf) + lane, ub);
                if (f.cnt < 0 && flag) *flag = 1;
                if (f.cnt == K) {
                    ch.d1 = f.d1;
                    ch.dk = f.dk;
                }
            }
        }
        __syncwarp();
    }
}

// Does a grid lie off the soundings (a hash of corner, cells and their side)?
__host__ __device__ inline bool grid_off(int32_t hx0, int32_t hy0, int32_t ncx, int32_t ncy, int32_t hash_cell,
                                         const GridView& g) {
    const int64_t x0 = (int64_t)g.x0 + g.cell / 2, y0 = (int64_t)g.y0 + g.cell / 2;
    const int64_t x1 = x0 + (int64_t)(g.nx - 1) * g.cell, y1 = y0 + (int64_t)(g.ny - 1) * g.cell;
    return x1 < hx0 || y1 < hy0 || x0 > hx0 + (int64_t)ncx * hash_cell || y0 > hy0 + (int64_t)ncy * hash_cell;
}
// Is the patch search the better one for a grid over this hash? Its staged list must
// hold the soundings of a patch and the radius around it (0.8 of it at the mean
// density; a patch of more costs a try and then its lanes' own searches), the
// bounds of its 32-bit arithmetic must hold, and the grid must not lie off the soundings
// (256 x 256 nodes 0.6 to 0.1 km off, IDW k = 32: 166 us by patches, 114 by threads;
// 6 km 216, 150).
template <int K>
__host__ __device__ inline bool knn_patch_fits(int64_t n_valid, int32_t hx0, int32_t hy0, int32_t ncx, int32_t ncy,
                                               int32_t hash_cell, const GridView& g) {
    if (n_valid <= 2 * K || g.cell >= kPatchMax / 7 || hash_cell > kCellMax) return false;
    if (grid_off(hx0, hy0, ncx, ncy, hash_cell, g)) return false;
    const double rho = (double)n_valid / ((double)ncx * (double)ncy * (double)hash_cell * (double)hash_cell);
    const double r = sqrt(KnnWarp<K>::kArea * K / (3.14159265 * rho)), c = hash_cell;
    const double w = (g.nx < 8 ? g.nx - 1 : 7) * (double)g.cell + 2 * r + c;
    const double t = (g.ny < 4 ? g.ny - 1 : 3) * (double)g.cell + 2 * r + c;
    return w * t * rho < 0.8 * KnnWarp<K>::CAP && 1.3 * r < kRadiusMax;
}
template <int K>
inline bool knn_patch_fits(const bg_soundings_info& s, const GridView& g) {
    return knn_patch_fits<K>(s.n_valid, s.bbox_x0_cm, s.bbox_y0_cm, s.ncx, s.ncy, s.cell_cm, g);
}
// Where patches do not serve: lanes of a warp for a node of the grid, or a thread? Off the
// soundings a lane's share of the records pays half as long (65,536 nodes k = 16 6 km
// off: 171 us by lanes, 100 by threads).
template <int K>
inline bool grid_by_lanes(const bg_soundings_info& s, const GridView& g, int64_t nodes) {
    return query_by_lanes<K>(grid_off(s.bbox_x0_cm, s.bbox_y0_cm, s.ncx, s.ncy, s.cell_cm, g) ? 2 * nodes : nodes);
}

// Does every bound over this grid fit a packed key? The farthest corner of the
// hash from any node bounds them all. Then no node is left to a wide pass, which
// saves a small call its flag and a launch (5 of 60 us).
inline bool packed_always(const HashView& h, const GridView& g) {
    const double x0 = (double)g.x0 + g.cell / 2, x1 = x0 + (double)(g.nx - 1) * g.cell;
    const double y0 = (double)g.y0 + g.cell / 2, y1 = y0 + (double)(g.ny - 1) * g.cell;
    const double hx1 = (double)h.hx0 + (double)h.ncx * h.cs, hy1 = (double)h.hy0 + (double)h.ncy * h.cs;
    const double dx = std::max(hx1 - x0, x1 - h.hx0), dy = std::max(hy1 - y0, y1 - h.hy0);
    return 1.001 * (dx * dx + dy * dy) + 2.0 < std::ldexp(1.0, 64 - h.idx_bits);
}

// Patches a warp takes along x: strips carry the radius from patch to patch,
// but leave enough warps for several waves.
inline int patch_strip_len(int64_t patches) {
    return (int)std::min<int64_t>(16, std::max<int64_t>(1, patches / (152 * 12 * 6)));
}

}  // namespace bg
