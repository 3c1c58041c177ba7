// Device code of fused k-NN + IDW, shared by the per-grid kernels (idw.cu)
// and the batched persistent kernels (batch.cu).
//
// Fused exact k-NN + inverse-distance weighting: a node per lane of a patch search
// (knn_warp.cuh), a query per half or whole warp (knn_query.cuh), or one per thread
// (knn.cuh).
//
// zhat = sum w_i z_i / sum w_i with w_i = d_i^-p over the k nearest valid
// soundings. It is evaluated as z_1 + sum w_i (z_i - z_1) / sum w_i with
// z_1 the nearest sounding's depth and w_i = (d_1^2 / d_i^2)^(p/2): the same
// quantity, but every term is an anomaly of a few metres (so only the final
// add rounds at ~3500 m) and every weight is in (0, 1]. The sums run in one
// fixed order over the ascending (d2, index) list (idw_tree8), so a node's
// result does not depend on the cell size, the launch shape, the kernel or
// what else runs.


#pragma once

#include <cmath>

#include "bg_internal.h"
#include "knn.cuh"
#include "knn_query.cuh"
#include "knn_warp.cuh"

namespace bg {


// d2 as float: a 32-bit conversion when it fits (64-bit ones use the FP64 pipe)
__device__ __forceinline__ float idw_d2f(uint64_t v) {
    return v < (1ull << 31) ? __int2float_rn((int)v) : __ull2float_rn(v);
}

// weight of a neighbour at squared distance di relative to the nearest (d1):
// (d1 / di)^(p/2), with l1 = log2(d1) and hp = p / 2
__device__ __forceinline__ float idw_weight(float d1, float l1, float hp, float power, float di) {
    if (power == 2.0f) return d1 / di;
    return exp2f(hp * (l1 - log2f(di)));
}

// The sums of an IDW run in one fixed order, so that every kernel that forms
// them gets bitwise the same depth: neighbour n >= 1 goes to partial n_t =
// (n - 1) mod 8, each partial adds its neighbours in ascending n, and the 8
// partials combine pairwise as ((p0 + p1) + (p2 + p3)) + ((p4 + p5) + (p6 +
// p7)). The kriging solve (2 threads per system, thread h holding the partials
// 4 h .. 4 h + 3) and the search by lanes (a lane per partial) form the same
// partials and combine them in that pattern.
constexpr int kIdwLanes = 8;

__device__ __forceinline__ float idw_tree8(const float (&p)[kIdwLanes]) {
    return ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
}

// IDW from keff neighbours in ascending (d2, index) order; get(i) returns
// (idw_d2f of the squared distance, depth) of the i-th.
template <class Get>
__device__ __forceinline__ float idw_sum(int keff, float power, Get get) {
    if (keff == 0) return __int_as_float(0x7fc00000);  // NaN: no valid sounding
    float d1, z1;
    get(0, d1, z1);
    if (d1 == 0.0f) return z1;  // node on top of a sounding
    float l1 = 0.0f;  // log2(d1), for powers other than 2
    if (power != 2.0f) l1 = log2f(d1);
    const float hp = 0.5f * power;
    float num[kIdwLanes], den[kIdwLanes];
#pragma unroll
    for (int q = 0; q < kIdwLanes; ++q) num[q] = den[q] = 0.0f;
    // eight neighbours per turn (one per partial), each model its own loop: short
    // enough to stay in the instruction cache beside a search
    auto turns = [&](auto weight) {
#pragma unroll 1
        for (int n0 = 1; n0 < keff; n0 += kIdwLanes) {
#pragma unroll
            for (int q = 0; q < kIdwLanes; ++q) {
                if (n0 + q >= keff) break;
                float di, zi;
                get(n0 + q, di, zi);
                const float w = weight(di);
                num[q] = fmaf(w, zi - z1, num[q]);
                den[q] += w;
            }
        }
    };
    if (power == 2.0f)
        turns([&](float d) { return idw_weight(d1, l1, hp, 2.0f, d); });
    else
        turns([&](float d) { return idw_weight(d1, l1, hp, power, d); });
    // neighbour 0 contributes weight 1 and anomaly 0
    return z1 + idw_tree8(num) / (1.0f + idw_tree8(den));
}

// The same with get(i) returning (d2, upload index).
template <class Get>
__device__ __forceinline__ float idw_from(const HashView& h, int keff, float power, Get get) {
    const int* zb = reinterpret_cast<const int*>(h.orig) + 2;  // z bits of record i at zb[4*i]
    return idw_sum(keff, power, [&](int n, float& d, float& z) {
        uint64_t d2;
        int i;
        get(n, d2, i);
        d = idw_d2f(d2);
        z = __int_as_float(__ldg(zb + 4 * (int64_t)i));
    });
}

// IDW of a node that the patch search served (knn_patch_row), and its k
// neighbours' upload indices to nbr, if any.
template <int K>
__device__ __forceinline__ void idw_served(const HashView& h, const typename KnnWarp<K>::Smem& sm, int ux, int uy,
                                           int k, float power, float* depth, int32_t* nbr) {
    const uint32_t* col = sm.buf + (threadIdx.x & 31);
    *depth = idw_sum(k, power, [&](int n, float& d, float& z) {
        const uint32_t q = col[n * 32] & kPlaceMask;
        const int4 c = sm.st[q];
        const int dx = c.x - ux, dy = c.y - uy;
        d = __int2float_rn(dx * dx + dy * dy);
        z = __int_as_float(__ldg(&h.rec[sm.pos[q]].z));
    });
    if (nbr)
        for (int n = 0; n < k; ++n) nbr[n] = __ldg(&h.rec[sm.pos[col[n * 32] & kPlaceMask]].w);
}
// The same of a node that it did not serve: a per-thread search, out of the way
// of the patch search's code.
template <int K>
__device__ __noinline__ KnnFar idw_lone(const HashView& h, int qx, int qy, uint64_t* hp, float ub, int k,
                                        float power, float* depth, int32_t* nbr) {
    const int cnt = knn_lane<K>(h, qx, qy, hp, ub);
    if (cnt < 0) return KnnFar{cnt, 0.0f, 0.0f};
    const int bits = h.idx_bits, keff = min(cnt, k);
    const uint64_t mask = (1ull << bits) - 1;
    *depth = idw_from(h, keff, power, [&](int n, uint64_t& dd, int& ii) {
        const uint64_t v = hp[n * 32];
        dd = v >> bits;
        ii = (int)(v & mask);
    });
    if (nbr) emit_ids<32>(nbr, hp, k, keff, mask);
    return knn_far<K>(h, hp, cnt);
}

// Wide-key IDW of one query point whose table bound does not fit the packed key
// (rare); others return.
template <int K>
__device__ __forceinline__ void idw_point_wide(const HashView& h, int qx, int qy, int k,
                                               float power, float* __restrict__ dout,
                                               int32_t* __restrict__ o) {
    if (!point_may_be_wide(h, qx, qy)) return;
    const Bound b = knn_bound<K>(h, qx, qy);
    if (packed_fits(h, b.tau0)) return;
    uint64_t d2[K];
    int id[K];
    const int keff = min(knn_scan_wide<K>(h, qx, qy, b, d2, id), k);
    *dout = idw_from(h, keff, power, [&](int i, uint64_t& dd, int& ii) {
        dd = d2[i];
        ii = id[i];
    });
    if (o)
        for (int i = 0; i < k; ++i) o[i] = i < keff ? id[i] : -1;
}

// IDW of the queries of a warp (knn_query): lane n of a query's G holds neighbour
// n, lanes 0 .. 7 the eight partial sums. valid: there is a query; ok: in range.
template <int G>
__device__ __forceinline__ void idw_query(const HashView& h, bool valid, bool ok, int qx, int qy, int k, float power,
                                          uint64_t* buf, float* depth, int32_t* nbr, int* flag) {
    const int lane = threadIdx.x & (G - 1);
    uint64_t key = 0;
    const int found = h.n_valid > 0 ? knn_query<G>(h, ok, qx, qy, k, buf, key) : 0, cnt = max(found, 0);
    const int u = lane < cnt ? (int)(key & ((1ull << h.idx_bits) - 1)) : -1;
    float d = 1.0f, z = 0.0f;
    if (u >= 0) {
        d = idw_d2f(key >> h.idx_bits);
        z = __int_as_float(__ldg(&h.orig[u].z));
    }
    const float d1 = __shfl_sync(kFull, d, 0, G), z1 = __shfl_sync(kFull, z, 0, G);
    float l1 = 0.0f;
    if (power != 2.0f) l1 = log2f(d1);
    const float w = idw_weight(d1, l1, 0.5f * power, power, d), dz = z - z1;
    float num = 0.0f, den = 0.0f;
    for (int n0 = 1; n0 < k; n0 += kIdwLanes) {
        const int n = n0 + (lane & 7);
        const float wn = __shfl_sync(kFull, w, n, G), dn = __shfl_sync(kFull, dz, n, G);
        if (n < cnt) {
            num = fmaf(wn, dn, num);
            den += wn;
        }
    }
#pragma unroll
    for (int s = 1; s < kIdwLanes; s *= 2) {
        num += __shfl_xor_sync(kFull, num, s);
        den += __shfl_xor_sync(kFull, den, s);
    }
    if (!valid) return;
    if (found < 0) {
        if (lane == 0 && flag) *flag = 1;
        return;
    }
    if (nbr && lane < k) nbr[lane] = u;
    if (lane == 0) *depth = cnt == 0 ? __int_as_float(0x7fc00000) : d1 == 0.0f ? z1 : z1 + num / (1.0f + den);
}

// Wide-key IDW of one grid node whose table bound does not fit the packed key
// (rare); others return.
template <int K>
__device__ __forceinline__ void idw_node_wide(const HashView& h, const GridView& g, int k, float power,
                                              float* __restrict__ depth, int32_t* __restrict__ nbr, NodeIdx nd) {
    if (nd.i >= g.nx || nd.j >= g.ny || h.n_valid == 0) return;
    const int64_t node = (int64_t)nd.j * g.nx + nd.i;
    const int qx = g.x0 + nd.i * g.cell + g.cell / 2;
    const int qy = g.y0 + nd.j * g.cell + g.cell / 2;
    const Bound b = knn_bound<K>(h, qx, qy);
    if (packed_fits(h, b.tau0)) return;
    uint64_t d2[K];
    int id[K];
    const int keff = min(knn_scan_wide<K>(h, qx, qy, b, d2, id), k);
    depth[node] = idw_from(h, keff, power, [&](int i, uint64_t& dd, int& ii) {
        dd = d2[i];
        ii = id[i];
    });
    if (nbr)
        for (int i = 0; i < k; ++i) nbr[node * k + i] = i < keff ? id[i] : -1;
}

}  // namespace bg
