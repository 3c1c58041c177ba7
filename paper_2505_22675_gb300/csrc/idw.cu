// Fused exact k-NN + inverse-distance weighting: per-grid kernels and launchers.
// The device code is in idw_dev.cuh.
#include <algorithm>

#include "idw_dev.cuh"
#include "knn_warp.cuh"

namespace bg {
namespace {

// Packed pass: one (16 * kLen) x 8 node patch per block, a strip of kLen
// nodes per thread (strip_len_for).
template <int K, int kLen>
__global__ void __launch_bounds__(128) k_idw(HashView h, GridView g, int k, float power,
                                             float* __restrict__ depth,
                                             int32_t* __restrict__ nbr, int* __restrict__ flag) {
    __shared__ uint64_t heap[K * 128];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gx = (g.nx + 16 * kLen - 1) / (16 * kLen);
    const NodeIdx o = strip_origin<kLen>(blockIdx.x % gx, blockIdx.x / gx, warp, lane);
    if (o.j >= g.ny) return;
    uint64_t* hp = heap + threadIdx.x;
    const int64_t row = (int64_t)o.j * g.nx;
    if (h.n_valid == 0) {
        for (int i = o.i; i < min(o.i + kLen, g.nx); ++i) {
            depth[row + i] = __int_as_float(0x7fc00000);
            if (nbr)
                for (int q = 0; q < k; ++q) nbr[(row + i) * k + q] = -1;
        }
        return;
    }
    const int bits = h.idx_bits;
    const uint64_t mask = (1ull << bits) - 1;
    auto emit = [&](int i, int cnt) {
        const int keff = min(cnt, k);
        depth[row + i] = idw_from(h, keff, power, [&](int q, uint64_t& dd, int& ii) {
            const uint64_t key = hp[q * 128];
            dd = key >> bits;
            ii = (int)(key & mask);
        });
        if (nbr) emit_ids<128>(nbr + (row + i) * k, hp, k, keff, mask);
    };
    knn_strip<128, decltype(emit), true, kLen>(h, g, K, o.i, o.j, hp, flag, emit);
}

// The same by patches of 8 x 4 nodes per warp (knn_warp.cuh), a strip of `len`
// patches along x each; spr strips per patch row.
template <int K>
__global__ void __launch_bounds__(64, KnnWarp<K>::kBlocksPerSM) k_idw_patch(HashView h, GridView g, int k, float power,
                                                  float* __restrict__ depth,
                                                  int32_t* __restrict__ nbr, int* __restrict__ flag,
                                                  int len, int spr) {
    __shared__ typename KnnWarp<K>::Smem smem[2];
    typename KnnWarp<K>::Smem& sm = smem[threadIdx.x >> 5];
    const unsigned w = blockIdx.x * 2 + (threadIdx.x >> 5);
    const int py = (int)(w / (unsigned)spr), p0 = (int)(w % (unsigned)spr) * len;
    if (py * 4 >= g.ny) return;
    auto out = [&](int i, int j) { return (int64_t)j * g.nx + i; };
    knn_patch_row<K>(
        h, g, sm, py * 4, g.ny, p0, p0 + len, flag,
        [&](int i, int j, int ux, int uy) {
            idw_served<K>(h, sm, ux, uy, k, power, depth + out(i, j), nbr ? nbr + out(i, j) * k : nullptr);
        },
        [&](int i, int j, int qx, int qy, uint64_t* hp, float ub) {
            return idw_lone<K>(h, qx, qy, hp, ub, k, power, depth + out(i, j), nbr ? nbr + out(i, j) * k : nullptr);
        });
}

// G lanes per query: points of a list or nodes of a grid. At most 56 registers (9 blocks):
// with the 64 that the compiler takes otherwise 2 % slower.
template <int G, class Queries>
__global__ void __launch_bounds__(32 * kQueryWarps, 9) k_idw_query(HashView h, Queries q, int64_t m, int k, float power,
                                                               float* __restrict__ depth,
                                                               int32_t* __restrict__ nbr, int* __restrict__ flag) {
    __shared__ uint64_t buf[32 * kQueryWarps * 2];
    const int n = threadIdx.x / G;
    const int64_t i = (int64_t)blockIdx.x * (32 * kQueryWarps / G) + n;
    int qx = h.hx0, qy = h.hy0;
    const bool ok = i < m && query_xy(q, i, qx, qy);
    idw_query<G>(h, i < m, ok, qx, qy, k, power, buf + n * 2 * G, depth + i, nbr ? nbr + i * k : nullptr, flag);
}

// Wide-key pass over the nodes the packed pass could not take; it returns at
// once when the packed pass flagged none.
template <int K>
__global__ void __launch_bounds__(128) k_idw_wide(HashView h, GridView g, int k, float power,
                                                  float* __restrict__ depth,
                                                  int32_t* __restrict__ nbr, int* __restrict__ flag) {
    if (*(volatile int*)flag == 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gx = (g.nx + 15) / 16;
    const int64_t nb = (int64_t)gx * ((g.ny + 7) / 8);
    for (int64_t b = blockIdx.x; b < nb; b += gridDim.x)
        idw_node_wide<K>(h, g, k, power, depth, nbr, patch_node((int)(b % gx), (int)(b / gx), warp, lane));
}

// d_flag: one int, or NULL to allocate one where it is needed
template <int K>
bg_status launch_k(const bg_soundings_s* s, const HashView& h, const GridView& g, int k, float power,
                   float* depth, int32_t* nbr, int* d_flag, cudaStream_t st, bg_ctx_s* prof_ctx) {
    const int64_t nb = (int64_t)((g.nx + 15) / 16) * ((g.ny + 7) / 8);
    const int len = strip_len_for((int64_t)g.nx * g.ny);
    const int64_t nbs = (int64_t)((g.nx + 16 * len - 1) / (16 * len)) * ((g.ny + 7) / 8);
    const int pnx = (g.nx + 7) / 8, pny = (g.ny + 3) / 4;
    const int plen = patch_strip_len((int64_t)pnx * pny), spr = (pnx + plen - 1) / plen;
    const bool wide = !packed_always(h, g);  // (an empty hash too: its nodes need no search)
    int* own = nullptr;
    if (!wide) d_flag = nullptr;
    if (wide && !d_flag) {
        const bg_status rc = dalloc(s->ctx, (void**)&own, sizeof(int), st);
        if (rc != BG_OK) return rc;
        d_flag = own;
    }
    cudaError_t e = wide ? cudaMemsetAsync(d_flag, 0, sizeof(int), st) : cudaSuccess;
    if (e == cudaSuccess) {
        ProfScope ps(prof_ctx, kProfIdw, (int64_t)g.nx * g.ny, st);
        if (knn_patch_fits<K>(s->info, g) && (int64_t)spr * pny < ((int64_t)1 << 31))
            k_idw_patch<K><<<(unsigned)(((int64_t)spr * pny + 1) / 2), 64, 0, st>>>(h, g, k, power, depth, nbr, d_flag,
                                                                                   plen, spr);
        else if (grid_by_lanes<K>(s->info, g, (int64_t)g.nx * g.ny))
            k_idw_query<query_lanes(K)><<<query_blocks<K>((int64_t)g.nx * g.ny), 32 * kQueryWarps, 0, st>>>(
                h, g, (int64_t)g.nx * g.ny, k, power, depth, nbr, d_flag);
        else if (len == 1)
            k_idw<K, 1><<<(unsigned)nbs, 128, 0, st>>>(h, g, k, power, depth, nbr, d_flag);
        else if (len == 2)
            k_idw<K, 2><<<(unsigned)nbs, 128, 0, st>>>(h, g, k, power, depth, nbr, d_flag);
        else
            k_idw<K, 4><<<(unsigned)nbs, 128, 0, st>>>(h, g, k, power, depth, nbr, d_flag);
    }
    if (wide && e == cudaSuccess)
        k_idw_wide<K><<<(unsigned)std::min<int64_t>(nb, 152 * 4), 128, 0, st>>>(h, g, k, power, depth, nbr, d_flag);
    note_launches(wide ? 2 : 1);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (own) dfree(s->ctx, own, sizeof(int), st);
    return e == cudaSuccess ? BG_OK : cuda_fail(e, "IDW launch");
}

// Query points: kLen consecutive points per thread (knn_chain).
template <int K, int kLen>
__global__ void __launch_bounds__(128) k_idw_pts(HashView h, PointsView q, int k, float power,
                                                 float* __restrict__ depth,
                                                 int32_t* __restrict__ nbr, int* __restrict__ flag) {
    __shared__ uint64_t heap[K * 128];
    const int64_t p0 = ((int64_t)blockIdx.x * 128 + threadIdx.x) * kLen;
    if (p0 >= q.m) return;
    uint64_t* hp = heap + threadIdx.x;
    const int bits = h.idx_bits;
    const uint64_t mask = (1ull << bits) - 1;
    auto none = [&](int64_t p) {
        depth[p] = __int_as_float(0x7fc00000);
        if (nbr)
            for (int i = 0; i < k; ++i) nbr[p * k + i] = -1;
    };
    if (h.n_valid == 0) {
        for (int64_t p = p0; p < min(p0 + kLen, q.m); ++p) none(p);
        return;
    }
    auto emit = [&](int64_t p, int cnt) {
        if (cnt < 0) {
            none(p);
            return;
        }
        const int keff = min(cnt, k);
        depth[p] = idw_from(h, keff, power, [&](int i, uint64_t& dd, int& ii) {
            const uint64_t key = hp[i * 128];
            dd = key >> bits;
            ii = (int)(key & mask);
        });
        if (nbr) emit_ids<128>(nbr + p * k, hp, k, keff, mask);
    };
    knn_chain<128, decltype(emit), kLen>(h, q.x, q.y, p0, q.m, K, hp, flag, emit);
}

template <int K>
__global__ void __launch_bounds__(128) k_idw_pts_wide(HashView h, PointsView q, int k, float power,
                                                      float* __restrict__ depth,
                                                      int32_t* __restrict__ nbr,
                                                      const int* __restrict__ flag) {
    if (flag && *(const volatile int*)flag == 0) return;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < q.m;
         p += (int64_t)gridDim.x * blockDim.x)
        idw_point_wide<K>(h, __ldg(q.x + p), __ldg(q.y + p), k, power, depth + p,
                          nbr ? nbr + p * k : nullptr);
}

template <int K>
bg_status launch_pts_k(const HashView& h, const PointsView& q, int k, float power, float* depth,
                       int32_t* nbr, cudaStream_t st, bg_ctx_s* prof_ctx) {
    const int len = strip_len_for(q.m);
    const int64_t threads = (q.m + len - 1) / len;
    const int64_t nb = (threads + 127) / 128;
    int* flag = nullptr;
    if (!query_by_lanes<K>(q.m)) {
        const bg_status rc = dalloc(prof_ctx, (void**)&flag, sizeof(int), st);
        if (rc != BG_OK) return rc;
    }
    cudaError_t e = flag ? cudaMemsetAsync(flag, 0, sizeof(int), st) : cudaSuccess;
    {
        ProfScope ps(prof_ctx, kProfIdw, q.m, st);
        if (query_by_lanes<K>(q.m))
            k_idw_query<query_lanes(K)><<<query_blocks<K>(q.m), 32 * kQueryWarps, 0, st>>>(
                h, q, q.m, k, power, depth, nbr, nullptr);
        else if (len == 1)
            k_idw_pts<K, 1><<<(unsigned)nb, 128, 0, st>>>(h, q, k, power, depth, nbr, flag);
        else if (len == 2)
            k_idw_pts<K, 2><<<(unsigned)nb, 128, 0, st>>>(h, q, k, power, depth, nbr, flag);
        else
            k_idw_pts<K, 4><<<(unsigned)nb, 128, 0, st>>>(h, q, k, power, depth, nbr, flag);
    }
    k_idw_pts_wide<K><<<(unsigned)std::min<int64_t>((q.m + 127) / 128, 152 * 4), 128, 0, st>>>(
        h, q, k, power, depth, nbr, flag);
    note_launches(2);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (flag) dfree(prof_ctx, flag, sizeof(int), st);
    return e == cudaSuccess ? BG_OK : cuda_fail(e, "IDW launch");
}

}  // namespace

bg_status launch_idw_points(const bg_soundings_s* s, const PointsView& q, int k, float power,
                            float* depth, int32_t* nbr, cudaStream_t st) {
    if (q.m == 0) return BG_OK;
    HashView h = s->h;
    const int K = k <= 4 ? 4 : k <= 8 ? 8 : k <= 16 ? 16 : 32;
    h.r0 = start_halfwidth(s, K);
    switch (K) {
        case 4: return launch_pts_k<4>(h, q, k, power, depth, nbr, st, s->ctx);
        case 8: return launch_pts_k<8>(h, q, k, power, depth, nbr, st, s->ctx);
        case 16: return launch_pts_k<16>(h, q, k, power, depth, nbr, st, s->ctx);
        default: return launch_pts_k<32>(h, q, k, power, depth, nbr, st, s->ctx);
    }
}

bg_status launch_idw(const bg_soundings_s* s, const GridView& g, int k, float power,
                     float* depth, int32_t* nbr, cudaStream_t st) {
    return launch_idw_with_flag(s, g, k, power, depth, nbr, nullptr, st);
}

bg_status launch_idw_with_flag(const bg_soundings_s* s, const GridView& g, int k, float power,
                               float* depth, int32_t* nbr, int* d_flag, cudaStream_t st) {
    HashView h = s->h;
    const int K = k <= 4 ? 4 : k <= 8 ? 8 : k <= 16 ? 16 : 32;
    h.r0 = start_halfwidth(s, K);
    switch (K) {
        case 4: return launch_k<4>(s, h, g, k, power, depth, nbr, d_flag, st, s->ctx);
        case 8: return launch_k<8>(s, h, g, k, power, depth, nbr, d_flag, st, s->ctx);
        case 16: return launch_k<16>(s, h, g, k, power, depth, nbr, d_flag, st, s->ctx);
        default: return launch_k<32>(s, h, g, k, power, depth, nbr, d_flag, st, s->ctx);
    }
}

}  // namespace bg
