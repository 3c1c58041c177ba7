// Exact k-nearest-neighbour search of one query by a whole warp, or by half of one
// where k <= 16 (two queries share the steps that few lanes take part in).
//
// For queries that share little of their neighbourhoods (points far apart, a
// grid of many soundings per node) there is nothing for a warp to stage once
// and scan 32 times, and a thread per query is a serial chain of some 100,000
// cycles (dependent loads, a heap in shared memory, lanes of unequal lengths)
// that a small list has nothing to hide behind. Here the lanes share the chain:
//   1. lane r counts the square of half-width r around the query's cell;
//   2. a lane per row of cells finds the row's run of records that can lie
//      within the bound;
//   3. the runs are one list of candidates, a lane each; those within the bound
//      (and below the k-th key so far) are collected in shared memory, and each
//      32 (16) of them are sorted across the lanes and merged into the best.
// The first bound is the radius that holds k + 2.5 sqrt(k) soundings at the
// square's density; with fewer than k inside, the scan runs again from the square's
// farthest corner, or in steps towards it where the square is large (query_wider).
// Keys and order are those of knn.cuh.
//
// Bound by instructions from about 10,000 queries on: 0.8 us for 1000 of them by
// halves of a warp, 1.3 by whole ones, most in 64-bit keys (sorting 32 takes 15
// exchanges of about 9).
#pragma once

#include "knn.cuh"

namespace bg {

constexpr int kQueryWarps = 4;  // warps a block
constexpr __host__ __device__ int query_lanes(int K) { return K <= 16 ? 16 : 32; }
template <int K>
inline unsigned query_blocks(int64_t m) {
    constexpr int n = 32 * kQueryWarps / query_lanes(K);
    return (unsigned)((m + n - 1) / n);
}

// Lanes per query, or a thread each? By threads 33 (k = 8), 52 (16), 80 us (32) go
// by whatever the number; by lanes 0.8 or 1.3 us a 1000. us, threads / lanes, IDW:
// 1,600 points k = 32 76 / 14, 6,000 nodes k = 32 130 / 20; holes of 5 % of a grid:
//   points      k = 8      k = 16      k = 32
//   30,000    34 / 31     52 / 31     82 / 51
//   45,000    35 / 41     55 / 41     90 / 74
//   60,000    35 / 49     55 / 52     99 / 95
//   80,000    36 / 60     56 / 64    117 / 124
// and of 1 %, where a thread's records are farther apart:
//   60,000    35 / 51     67 / 61    158 / 107
//   80,000    47 / 65     78 / 76    181 / 131    (k = 16, ids 92 / 72)
// The line of k = 16 lies where the sparse lists gain what the dense ones lose.
template <int K>
inline bool query_by_lanes(int64_t m) {
    return m <= (K <= 8 ? 152 * 224 : K == 16 ? 152 * 576 : 152 * 384);
}

// G lanes (16 or 32) work on a query; both halves of a warp take every step
// together, so a half that has finished repeats or idles until the other has.
template <int G>
__device__ __forceinline__ unsigned query_ballot(bool v) {
    const unsigned m = __ballot_sync(kFull, v);
    if constexpr (G == 32) return m;
    return m >> (threadIdx.x & 16) & 0xffffu;
}
template <int G>
__device__ __forceinline__ int query_max(int v) {  // over the queries of a warp
    return G == 32 ? v : max(v, __shfl_xor_sync(kFull, v, 16));
}
__device__ __forceinline__ uint64_t query_pick(uint64_t x, int stride, bool smaller) {
    const uint64_t y = __shfl_xor_sync(kFull, x, stride);
    return (y < x) == smaller ? y : x;
}
// ascending over the G lanes
template <int G>
__device__ __forceinline__ uint64_t query_sort(uint64_t x, int lane) {
#pragma unroll
    for (int size = 2; size <= G; size *= 2)
#pragma unroll
        for (int s = size / 2; s > 0; s /= 2) x = query_pick(x, s, ((lane & s) == 0) == ((lane & size) == 0));
    return x;
}
// the G smallest of two ascending sequences, ascending
template <int G>
__device__ __forceinline__ uint64_t query_merge(uint64_t a, uint64_t b, int lane) {
    const uint64_t r = __shfl_xor_sync(kFull, b, G - 1);
    uint64_t x = r < a ? r : a;
#pragma unroll
    for (int s = G / 2; s > 0; s /= 2) x = query_pick(x, s, (lane & s) == 0);
    return x;
}

// How far (cm, rounded down) a query x, y from the hash's origin lies outside of the hash.
__device__ __forceinline__ float query_outside(int64_t x, int64_t y, int cs, int ncx, int ncy) {
    const float ox = (float)max(max(-x, x - ((int64_t)ncx * cs - 1)), (int64_t)0);
    const float oy = (float)max(max(-y, y - ((int64_t)ncy * cs - 1)), (int64_t)0);
    return 0.99999f * sqrtf(ox * ox + oy * oy);
}

// The squared bound to try after one of tau has held fewer than kc: the part of its radius
// past the distance that the kc-th can have at least is doubled, up to tau0. The
// square of half-width lo cells around the query's cell holds fewer than kc, the next one
// count. Out of the way: a miss is rare where soundings lie all around. The farthest
// corner at once costs a query off to one side most of what lies within its reach: 21,845
// points k = 8, half of them up to 250 m from the soundings, 673 us; so 89, by threads
// 185.
static __device__ __noinline__ int64_t query_wider(int64_t x, int64_t y, int cs, int ncx, int ncy, int lo, int count, int kc,
                                            int64_t tau, int64_t tau0) {
    const int cx = (int)min(max(x / cs, (int64_t)0), (int64_t)ncx - 1), cy = (int)min(max(y / cs, (int64_t)0), (int64_t)ncy - 1);
    int64_t d = LLONG_MAX;
    if (cx - lo > 0) d = min(d, x - (int64_t)(cx - lo) * cs);
    if (cx + lo < ncx - 1) d = min(d, (int64_t)(cx + lo + 1) * cs - x);
    if (cy - lo > 0) d = min(d, y - (int64_t)(cy - lo) * cs);
    if (cy + lo < ncy - 1) d = min(d, (int64_t)(cy + lo + 1) * cs - y);
    const float in = lo < 0 || d == LLONG_MAX ? 0.0f : 0.99999f * (float)max(d, (int64_t)0);
    const float near = fmaxf(in, query_outside(x, y, cs, ncx, ncy)), c = (float)cs;
    float past = sqrtf((float)tau) - near;
    if (past <= 0.0f) {
        // soundings on one side only: they begin in the ring of cells between the two squares;
        // past it by the height of the circle's segment that holds kc + 2.5 sqrt(kc) at
        // the density of one side of the ring
        const float want = (float)kc + 2.5f * sqrtf((float)kc), side = (float)(2 * lo + 3) * c * c;
        past = c + __powf(0.75f * want * side / ((float)max(count, 1) * sqrtf(2.0f * near)), 0.6666667f);
    } else {
        past = 2.0f * past + 0.5f * c;
    }
    const float r = near + past;
    // (a 64th more at least: the steps end whatever the rounding)
    return min(tau0, r * r < 0.64f * (float)tau0 ? max((int64_t)(r * r), tau + tau / 64 + 1) : tau0);
}

// The kc (<= G) nearest of (qx, qy), the same in every lane of the query: lane n
// gets the n-th packed key; returns how many there are (0 unless ok), or -1 where
// the bound does not fit a packed key. buf: 2 G keys of the query's own.
// h.n_valid > 0; all lanes of the warp.
template <int G>
__device__ __forceinline__ int knn_query(const HashView& h, bool ok, int qx, int qy, int kc, uint64_t* buf,
                                         uint64_t& best) {
    const int lane = threadIdx.x & (G - 1), bits = h.idx_bits;
    const int cx = clamp_cell(h, (int64_t)qx - h.hx0, h.ncx);
    const int cy = clamp_cell(h, (int64_t)qy - h.hy0, h.ncy);
    const int rmax = max(max(cx, h.ncx - 1 - cx), max(cy, h.ncy - 1 - cy));
    // smallest half-width of kc soundings (rmax: the whole hash): lo too small, hi not
    int lo = -1, hi = rmax, r = min(lane, rmax), count;
    for (;;) {
        const int c = sat_count(h, max(cx - r, 0), max(cy - r, 0), min(cx + r, h.ncx - 1), min(cy + r, h.ncy - 1));
        const unsigned m = query_ballot<G>(c >= kc || r == hi);
        const int j = m ? __ffs(m) - 1 : G;
        const int below = __shfl_sync(kFull, r, max(j - 1, 0), G), at = __shfl_sync(kFull, r, j, G);
        count = __shfl_sync(kFull, c, j, G);
        if (j > 0) lo = below;
        if (j < G) hi = at;
        if (__all_sync(kFull, j < G && hi - lo <= 1)) break;  // (the same again where this holds already)
        const int w = (hi - lo + G - 1) / G;  // the last lane reaches hi, which counts as enough
        r = min(lo + w * (lane + 1), hi);
    }
    int64_t tau0, tau;
    bool fits;
    {
        const int xa = max(cx - hi, 0), xb = min(cx + hi, h.ncx - 1);
        const int ya = max(cy - hi, 0), yb = min(cy + hi, h.ncy - 1);
        const int64_t xlo = (int64_t)h.hx0 + (int64_t)xa * h.cs, xhi = (int64_t)h.hx0 + (int64_t)(xb + 1) * h.cs - 1;
        const int64_t ylo = (int64_t)h.hy0 + (int64_t)ya * h.cs, yhi = (int64_t)h.hy0 + (int64_t)(yb + 1) * h.cs - 1;
        const int64_t mdx = max((int64_t)qx - xlo, xhi - (int64_t)qx), mdy = max((int64_t)qy - ylo, yhi - (int64_t)qy);
        tau0 = tau = mdx * mdx + mdy * mdy;
        fits = packed_fits(h, tau0);
        const float fk = (float)kc;
        const float tg = (fk + 2.5f * sqrtf(fk)) * (float)(xhi - xlo + 1) * (float)(yhi - ylo + 1) /
                         (3.14159265f * (float)count);
        if (count >= kc && tg < (float)tau0) tau = (int64_t)tg;
    }
    const bool scans = ok && fits;
    if (!scans) tau = tau0 = 0;
    const int64_t xmin = h.hx0, xmax = (int64_t)h.hx0 + (int64_t)h.ncx * h.cs - 1;
    for (;;) {
        uint64_t thr = (uint64_t)(tau + 1) << bits;
        int np = 0;
        bool some = false;
        auto flush = [&](uint64_t x) {
            x = query_sort<G>(x, lane);
            best = some ? query_merge<G>(best, x, lane) : x;
            some = true;
            thr = min(thr, __shfl_sync(kFull, best, kc - 1, G));
        };
        best = ~0ull;
        const int64_t rad = isqrt_ub(tau);
        const int rlo = clamp_cell(h, qy - rad - h.hy0, h.ncy);
        const int rhi = scans ? clamp_cell(h, qy + rad - h.hy0, h.ncy) : -1;
        const int turns = query_max<G>(scans ? (rhi - rlo) / G + 1 : 0);
        for (int t = 0; t < turns; ++t) {
            const int row = rlo + t * G + lane;
            int s = 0, len = 0;
            if (row <= rhi) {
                const int64_t ylo = (int64_t)h.hy0 + (int64_t)row * h.cs, yhi = ylo + h.cs - 1;
                const int64_t dy = qy < ylo ? ylo - qy : (qy > yhi ? qy - yhi : 0);
                if (dy * dy <= tau) {
                    const int64_t dxm = isqrt_ub(tau - dy * dy);
                    const int64_t xa = max((int64_t)qx - dxm, xmin), xb = min((int64_t)qx + dxm, xmax);
                    if (xa <= xb) {
                        const int32_t* cs = h.cell_start + (int64_t)row * h.ncx;
                        s = __ldg(cs + cell_of(h, xa - h.hx0));
                        len = __ldg(cs + cell_of(h, xb - h.hx0) + 1) - s;
                    }
                }
            }
            int off = len;  // inclusive prefix
#pragma unroll
            for (int d = 1; d < G; d *= 2) {
                const int o = __shfl_up_sync(kFull, off, d, G);
                if (lane >= d) off += o;
            }
            const int total = __shfl_sync(kFull, off, G - 1, G), most = query_max<G>(total);
            off -= len;
            const int rel = s - off;
            for (int b = 0; b < most; b += G) {
                const int i = b + lane;
                int w = 0;  // the last row that starts at or before candidate i
#pragma unroll
                for (int d = G / 2; d > 0; d /= 2)
                    if (__shfl_sync(kFull, off, w + d, G) <= i) w += d;
                const int p = i + __shfl_sync(kFull, rel, w, G);
                uint64_t key = ~0ull;
                if (i < total) {
                    const int4 v = __ldg(h.rec + p);
                    const int dx = v.x - qx, dy = v.y - qy;
                    const uint64_t d2 = (uint64_t)((long long)dx * dx + (long long)dy * dy);
                    const uint64_t c = (d2 << bits) | (uint32_t)v.w;
                    if (d2 <= (uint64_t)tau && c < thr) key = c;
                }
                const unsigned m = query_ballot<G>(key != ~0ull);
                if (key != ~0ull) buf[np + __popc(m & ((1u << lane) - 1))] = key;
                np += __popc(m);
                if (__any_sync(kFull, np >= G)) {  // a query that has fewer sorts what it has
                    __syncwarp();
                    const uint64_t x = lane < np ? buf[lane] : ~0ull, rest = buf[G + lane];
                    __syncwarp();
                    np = max(np - G, 0);
                    if (lane < np) buf[lane] = rest;
                    flush(x);
                }
            }
        }
        if (__any_sync(kFull, np > 0)) {
            __syncwarp();
            const uint64_t x = lane < np ? buf[lane] : ~0ull;
            __syncwarp();
            flush(x);
        }
        const int cnt = min(kc, __popc(query_ballot<G>(best != ~0ull)));
        const bool more = cnt < kc && tau != tau0;
        if (!__any_sync(kFull, more)) return ok && !fits ? -1 : cnt;
        if (more) {  // (a few cells hold enough: their corner)
            if (lo <= 1)
                tau = tau0;
            else
                tau = query_wider((int64_t)qx - h.hx0, (int64_t)qy - h.hy0, h.cs, h.ncx, h.ncy, lo, count, kc, tau, tau0);
        }
    }
}

// The i-th query of a launch: a point of a list (false: out of range), or a
// node of a grid.
__device__ __forceinline__ bool query_xy(const PointsView& q, int64_t i, int& x, int& y) {
    x = __ldg(q.x + i);
    y = __ldg(q.y + i);
    return query_in_range(x, y);
}
__device__ __forceinline__ bool query_xy(const GridView& g, int64_t i, int& x, int& y) {
    const int64_t j = i < ((int64_t)1 << 32) ? (int64_t)((uint32_t)i / (uint32_t)g.nx) : i / g.nx;
    x = g.x0 + (int)(i - j * g.nx) * g.cell + g.cell / 2;
    y = g.y0 + (int)j * g.cell + g.cell / 2;
    return true;
}

}  // namespace bg
