// Local ordinary kriging (Sec. III-C): the per-grid kernels and their launcher.
// The device code (k-NN to ids, reduced-system assembly, Cholesky, refinement)
// is in okrige_dev.cuh; see there for the formulation.
#include <algorithm>

#include "okrige_dev.cuh"

namespace bg {
namespace {

// grid rows [j0, j1); j0 is a multiple of 8; a strip of kLen nodes per thread
// (strip_len_for). 64-thread blocks: the 16 KB heap (K = 32) plus the
// per-block reserve lets 13 blocks (26 warps) share an SM, against 6 blocks
// (24 warps) of 128.
template <int K, int kLen>
__global__ void __launch_bounds__(64) k_knn_ids(HashView h, GridView g, int k, int j0, int j1,
                                                int32_t* __restrict__ ids, int* __restrict__ flag) {
    __shared__ uint64_t heap[K * 64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gx = (g.nx + 16 * kLen - 1) / (16 * kLen);
    // (16 * kLen) x 4 node patches: warp w covers columns w * 8 * kLen ..
    const int px = blockIdx.x % gx, py = j0 / 4 + blockIdx.x / gx;
    const NodeIdx o{px * 16 * kLen + warp * 8 * kLen + (lane & 7) * kLen, py * 4 + (lane >> 3)};
    if (o.j >= j1) return;
    uint64_t* hp = heap + threadIdx.x;
    int32_t* base = ids + ((int64_t)(o.j - j0) * g.nx) * k;
    if (h.n_valid == 0) {
        for (int i = o.i; i < min(o.i + kLen, g.nx); ++i)
            for (int q = 0; q < k; ++q) base[(int64_t)i * k + q] = -1;
        return;
    }
    const uint64_t mask = (1ull << h.idx_bits) - 1;
    // k == K (a multiple of 4) puts every node's ids on a 16-byte boundary when
    // the buffer is aligned: a full heap is then drained straight into them,
    // four ids per store; otherwise it is sorted in place and copied out
    const bool vec = k == K && K % 4 == 0 && (reinterpret_cast<uintptr_t>(ids) & 15) == 0;
    auto emit = [&](int i, int cnt) {
        int32_t* out = base + (int64_t)i * k;
        if (vec && cnt == K) {
            drain_ids<K, 64>(out, hp, mask);
            return;
        }
        for (int e = cnt - 1; e > 0; --e) {  // heapsort of a partial heap
            const uint64_t v = hp[e * 64];
            hp[e * 64] = hp[0];
            heap_sift_down<64>(hp, 0, e, v);
        }
        emit_ids<64>(out, hp, k, cnt, mask);
    };
    knn_strip<64, decltype(emit), false, kLen>(h, g, K, o.i, o.j, hp, flag, emit);
}

// The same by patches of 8 x 4 nodes per warp (knn_warp.cuh), a strip of `len`
// patches along x each, spr strips per patch row, into either layout.
template <int K>
__global__ void __launch_bounds__(64, KnnWarp<K>::kBlocksPerSM) k_knn_ids_patch(HashView h, GridView g, int k,
                                                                                IdsView ids,
                                                                                int* __restrict__ flag, int len,
                                                                                int spr) {
    __shared__ typename KnnWarp<K>::Smem smem[2];
    typename KnnWarp<K>::Smem& sm = smem[threadIdx.x >> 5];
    const unsigned w = blockIdx.x * 2 + (threadIdx.x >> 5);
    const int py = (int)(w / (unsigned)spr), p0 = (int)(w % (unsigned)spr) * len;
    const int jb = ids.j0 + py * 4;
    if (jb >= ids.j1) return;
    auto slot = [&](int i, int j) {
        return ids.p + (ids.stride > 0 ? node_slot(ids, i, j) : ((int64_t)(j - ids.j0) * g.nx + i) * k);
    };
    knn_patch_row<K>(
        h, g, sm, jb, ids.j1, p0, p0 + len, flag,
        [&](int i, int j, int, int) { ids_served<K>(h, sm, k, slot(i, j), ids.stride); },
        [&](int i, int j, int qx, int qy, uint64_t* hp, float ub) {
            return ids_lone<K>(h, qx, qy, hp, ub, k, slot(i, j), ids.stride);
        });
}

// The ids of queries i0 .. i0 + m - 1, G lanes each (put_point_id).
template <int G, class Queries>
__global__ void __launch_bounds__(32 * kQueryWarps, 9) k_knn_ids_query(HashView h, Queries q, int64_t i0, int64_t m, int k,
                                                                   int32_t* __restrict__ ids, int64_t stride,
                                                                   int* __restrict__ flag) {
    __shared__ uint64_t buf[32 * kQueryWarps * 2];
    const int n = threadIdx.x / G, lane = threadIdx.x & (G - 1);
    const int64_t i = (int64_t)blockIdx.x * (32 * kQueryWarps / G) + n;
    int qx = h.hx0, qy = h.hy0;
    const bool ok = i < m && query_xy(q, i0 + i, qx, qy);
    uint64_t key = 0;
    const int cnt = h.n_valid > 0 ? knn_query<G>(h, ok, qx, qy, k, buf + n * 2 * G, key) : 0;
    if (i >= m) return;
    if (cnt < 0) {
        if (lane == 0 && flag) *flag = 1;
    } else if (lane < k) {
        put_point_id(ids + i * (stride > 0 ? 1 : k), stride, lane,
                     lane < cnt ? (int)(key & ((1ull << h.idx_bits) - 1)) : -1);
    }
}

template <int K>
__global__ void __launch_bounds__(128) k_knn_ids_wide(HashView h, GridView g, int k, IdsView ids,
                                                      int* __restrict__ flag) {
    if (*(volatile int*)flag == 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gx = (g.nx + 15) / 16;
    const int64_t nb = (int64_t)gx * ((ids.j1 - ids.j0 + 7) / 8);
    for (int64_t b = blockIdx.x; b < nb; b += gridDim.x)
        knn_ids_node_wide<K>(h, g, k, ids, patch_node((int)(b % gx), ids.j0 / 8 + (int)(b / gx), warp, lane));
}

// Solve blocks take `per` consecutive batches of 128 systems: one take of the
// tensor memory and one block start (a twentieth of a batch) for several, in at
// least four rounds of blocks, so that small grids spread over the SMs. Of those
// the count whose rounds add up to the fewest batches: a last round of which
// most blocks are missing takes as long as a whole one (16,262 batches over 152
// places: 14 rounds of 8 2575 us, 27 of 4 2511, 107 of 1 2589; 1,639: 6 rounds of
// 2 305 us, 11 of 1 289).
template <int K>
int solve_batches_per_block(int64_t batches) {
    const int64_t places = 152 * Geo<K>::BLOCKS;
    int best = 1;
    double least = 1e300;
    for (int per = 1; per <= 8 && (per == 1 || batches >= 4 * places * per); ++per) {
        const int64_t blocks = (batches + per - 1) / per, rounds = (blocks + places - 1) / places;
        const double t = (double)rounds * (per + 0.05);
        if (t < least) {
            least = t;
            best = per;
        }
    }
    return best;
}

template <int K, class Fn>
__device__ __forceinline__ void solve_batches(const IdsView& ids, int64_t nsys, int k, int per, Fn fn) {
    __shared__ uint32_t slot;
    const uint32_t tm = tmem_take<Geo<K>::COLS>(&slot);
    const int64_t batches = (nsys + kSolveSystems - 1) / kSolveSystems;
    const int64_t b0 = (int64_t)blockIdx.x * per, b1 = min(b0 + per, batches);
    // the ids of this block's other batches and of the block that will follow it
    // on its SM: the k-NN kernel wrote them a launch ago and they have left L2
    // since
    for (int64_t b = b0 + 1; b < b1; ++b) prefetch_ids_l2(ids, nsys, k, b);
    prefetch_ids_l2(ids, nsys, k, b0 + (int64_t)152 * Geo<K>::BLOCKS * per);
    fn(b0, b1, tm);
    tmem_give<Geo<K>::COLS>(&slot);
}

// dynamic shared memory: Geo<K>::SMEM bytes
template <int K, bool kSph, bool kIdw>
__global__ void __launch_bounds__(Geo<K>::THREADS, Geo<K>::BLOCKS) k_okrige_solve(
    HashView h, GridView g, int k, OkParams p, int64_t node0, int64_t nsys, IdsView ids,
    float* __restrict__ depth, float* __restrict__ var, IdwFuse fz, int per) {
    extern __shared__ __align__(16) float4 smem[];
    solve_batches<K>(ids, nsys, k, per, [&](int64_t b0, int64_t b1, uint32_t tm) {
        okrige_solve_range<K, kSph, false, kIdw>(h, g, k, p, node0, nsys, ids, depth, var, b0, b1, smem,
                                                 tm, nullptr, nullptr, fz);
    });
}

// Copy rows [off, off + n) of the outputs to their host destinations on
// ho->cs, after the work enqueued so far on st.
bg_status copy_rows_to_host(const HostOut* ho, int64_t off, int64_t n, const float* idw,
                            const float* depth, const float* var, cudaStream_t st) {
    cudaError_t e = cudaEventRecord(ho->ev, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(ho->cs, ho->ev, 0);
    const size_t bytes = (size_t)n * sizeof(float);
    if (e == cudaSuccess && ho->idw && idw)
        e = cudaMemcpyAsync(ho->idw + off, idw + off, bytes, cudaMemcpyDeviceToHost, ho->cs);
    if (e == cudaSuccess && ho->depth)
        e = cudaMemcpyAsync(ho->depth + off, depth + off, bytes, cudaMemcpyDeviceToHost, ho->cs);
    if (e == cudaSuccess && ho->var && var)
        e = cudaMemcpyAsync(ho->var + off, var + off, bytes, cudaMemcpyDeviceToHost, ho->cs);
    return e == cudaSuccess ? BG_OK : cuda_fail(e, "device-to-host copy");
}

template <int K, bool kSph>
bg_status launch_k(const bg_soundings_s* snd, const HashView& h, const GridView& g, int k, const OkParams& p, float* depth,
                   float* var, int32_t* nbr, bg_ctx_s* ctx, cudaStream_t st, const IdwFuse* fz,
                   const HostOut* ho) {
    using Gm = Geo<K>;
    // grid rows per chunk: the id buffer stays near 1 GiB. The patch search writes the
    // patches layout where its rounding up to whole patches costs little
    // (slots_pay) and, under a budget, no memory; else the rows layout, as the
    // per-thread search always does. With lists the caller's nbr_out is the (whole)
    // buffer: a call that brings one takes no memory for another.
    const auto chunk_rows = [&](int64_t width) {
        const int64_t most = ((((int64_t)1 << 28) / (k * width)) / 8) * 8;
        return std::min<int64_t>(g.ny, std::max<int64_t>(8, most));
    };
    const size_t flag_bytes = 256;
    const int pnx = (g.nx + 7) / 8;
    int64_t rows = chunk_rows((int64_t)pnx * 8);
    const int64_t slots = (int64_t)pnx * ((rows + 3) / 4) * 32;
    const bool patches = knn_patch_fits<K>(snd->info, g);
    bool slot_ids = patches && !nbr && (ctx->budget ? slots <= rows * g.nx : slots_pay(slots, rows * g.nx));
    size_t id_bytes = 0;
    void* scratch = nullptr;
    bg_status rc = BG_OK;
    if (slot_ids) {
        id_bytes = (size_t)slots * k * sizeof(int32_t);
        rc = dalloc(ctx, &scratch, flag_bytes + id_bytes, st);
        if (rc == BG_ERR_CUDA) cudaGetLastError();  // a full device: the rows layout needs less
        slot_ids = rc == BG_OK;
    }
    if (!slot_ids) {
        rows = nbr ? g.ny : chunk_rows(g.nx);
        id_bytes = nbr ? 0 : (size_t)rows * g.nx * k * sizeof(int32_t);
        rc = dalloc(ctx, &scratch, flag_bytes + id_bytes, st);
    }
    if (rc != BG_OK) return rc;
    const bool wide = !packed_always(h, g);
    int* flag = (int*)scratch;
    const int gx = (g.nx + 15) / 16;
    cudaError_t ea = cudaFuncSetAttribute(k_okrige_solve<K, kSph, false>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, Gm::SMEM);
    if constexpr (K == 32)
        if (ea == cudaSuccess)
            ea = cudaFuncSetAttribute(k_okrige_solve<K, kSph, true>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, Gm::SMEM);
    if (ea != cudaSuccess) {
        dfree(ctx, scratch, flag_bytes + id_bytes, st);
        return cuda_fail(ea, "solve shared-memory size");
    }
    for (int64_t j0 = 0; j0 < g.ny; j0 += rows) {
        const int64_t j1 = std::min<int64_t>(g.ny, j0 + rows);
        const int64_t nb = (int64_t)gx * ((j1 - j0 + 7) / 8);
        const int len = strip_len_for((j1 - j0) * (int64_t)g.nx);
        const int64_t nbs = (int64_t)((g.nx + 16 * len - 1) / (16 * len)) * ((j1 - j0 + 3) / 4);
        int32_t* chunk_ids = nbr ? nbr + j0 * g.nx * k : (int32_t*)((char*)scratch + flag_bytes);
        cudaError_t e = wide ? cudaMemsetAsync(flag, 0, sizeof(int), st) : cudaSuccess;
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "memset");
            break;
        }
        const int64_t nodes = (j1 - j0) * g.nx;
        const int pny = (int)((j1 - j0 + 3) / 4);
        const IdsView ids{chunk_ids, slot_ids ? slots : 0, pnx, (int)j0, (int)j1};
        const int64_t nsys = slot_ids ? (int64_t)pnx * pny * 32 : nodes;
        {
            ProfScope ps(ctx, kProfKnnIds, nodes, st);
            const int plen = patch_strip_len((int64_t)pnx * pny), spr = (pnx + plen - 1) / plen;
            if (patches)
                k_knn_ids_patch<K><<<(unsigned)(((int64_t)spr * pny + 1) / 2), 64, 0, st>>>(
                    h, g, k, ids, flag, plen, spr);
            else if (grid_by_lanes<K>(snd->info, g, nodes))
                k_knn_ids_query<query_lanes(K)><<<query_blocks<K>(nodes), 32 * kQueryWarps, 0, st>>>(
                    h, g, j0 * g.nx, nodes, k, chunk_ids, 0, flag);
            else if (len == 1)
                k_knn_ids<K, 1><<<(unsigned)nbs, 64, 0, st>>>(h, g, k, (int)j0, (int)j1, chunk_ids, flag);
            else if (len == 2)
                k_knn_ids<K, 2><<<(unsigned)nbs, 64, 0, st>>>(h, g, k, (int)j0, (int)j1, chunk_ids, flag);
            else
                k_knn_ids<K, 4><<<(unsigned)nbs, 64, 0, st>>>(h, g, k, (int)j0, (int)j1, chunk_ids, flag);
        }
        if (wide)
            k_knn_ids_wide<K><<<(unsigned)std::min<int64_t>(nb, 152 * 4), 128, 0, st>>>(
                h, g, k, ids, flag);
        note_launches(wide ? 3 : 2);
        const int64_t batches = (nsys + kSolveSystems - 1) / kSolveSystems;
        const int per = solve_batches_per_block<K>(batches);
        const unsigned sb = (unsigned)((batches + per - 1) / per);
        {
            ProfScope ps(ctx, kProfSolve, nodes, st);
            bool fused = false;
            if constexpr (K == 32) {
                if (fz) {
                    k_okrige_solve<K, kSph, true><<<sb, Gm::THREADS, Gm::SMEM, st>>>(
                        h, g, k, p, j0 * g.nx, nsys, ids, depth, var, *fz, per);
                    fused = true;
                }
            }
            if (!fused)
                k_okrige_solve<K, kSph, false><<<sb, Gm::THREADS, Gm::SMEM, st>>>(
                    h, g, k, p, j0 * g.nx, nsys, ids, depth, var, IdwFuse{}, per);
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "kriging launch");
            break;
        }
        if (ho) {
            rc = copy_rows_to_host(ho, j0 * g.nx, nodes, fz ? fz->out : nullptr, depth, var, st);
            if (rc != BG_OK) break;
        }
    }
    if (ho && rc == BG_OK) {  // later work on st waits for the last copy
        cudaError_t e = cudaEventRecord(ho->ev, ho->cs);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ho->ev, 0);
        if (e != cudaSuccess) rc = cuda_fail(e, "copy-stream join");
    }
    dfree(ctx, scratch, flag_bytes + id_bytes, st);
    return rc;
}

// ------------------------------------------------------------ query points

// points [p0, p1), kLen consecutive points per thread (strip_len_for)
template <int K, int kLen>
__global__ void __launch_bounds__(128) k_knn_ids_pts(HashView h, PointsView q, int k, int64_t p0,
                                                     int64_t p1, int32_t* __restrict__ ids, int64_t stride,
                                                     int* __restrict__ flag) {
    __shared__ uint64_t heap[K * 128];
    const int64_t a = p0 + ((int64_t)blockIdx.x * 128 + threadIdx.x) * kLen;
    if (a >= p1) return;
    uint64_t* hp = heap + threadIdx.x;
    if (h.n_valid == 0) {
        for (int64_t p = a; p < min(a + kLen, p1); ++p)
            for (int i = 0; i < k; ++i) put_point_id(ids + (p - p0) * (stride > 0 ? 1 : k), stride, i, -1);
        return;
    }
    const uint64_t mask = (1ull << h.idx_bits) - 1;
    auto emit = [&](int64_t p, int cnt) {
        if (stride > 0)
            for (int i = 0; i < k; ++i)
                put_point_id(ids + (p - p0), stride, i, i < cnt ? (int)(hp[i * 128] & mask) : -1);
        else
            emit_ids<128>(ids + (p - p0) * k, hp, k, cnt, mask);
    };
    knn_chain<128, decltype(emit), kLen>(h, q.x, q.y, a, p1, K, hp, flag, emit);
}

template <int K>
__global__ void __launch_bounds__(128) k_knn_ids_pts_wide(HashView h, PointsView q, int k,
                                                          int64_t p0, int64_t p1,
                                                          int32_t* __restrict__ ids, int64_t stride,
                                                          const int* __restrict__ flag) {
    if (flag && *(const volatile int*)flag == 0) return;
    for (int64_t p = p0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < p1;
         p += (int64_t)gridDim.x * blockDim.x)
        knn_ids_point_wide<K>(h, __ldg(q.x + p), __ldg(q.y + p), k, ids + (p - p0) * (stride > 0 ? 1 : k), stride);
}

// dynamic shared memory: Geo<K>::SMEM bytes
template <int K, bool kSph>
__global__ void __launch_bounds__(Geo<K>::THREADS, Geo<K>::BLOCKS) k_okrige_solve_pts(
    HashView h, PointsView q, int k, OkParams p, int64_t p0, int64_t nsys, IdsView ids,
    float* __restrict__ depth, float* __restrict__ var, int per) {
    extern __shared__ __align__(16) float4 smem[];
    solve_batches<K>(ids, nsys, k, per, [&](int64_t b0, int64_t b1, uint32_t tm) {
        okrige_solve_range<K, kSph, true, false>(h, GridView{}, k, p, p0, nsys, ids, depth, var, b0, b1,
                                                 smem, tm, q.x, q.y);
    });
}

template <int K, bool kSph>
bg_status launch_pts_k(const HashView& h, const PointsView& q, int k, const OkParams& p,
                       float* depth, float* var, int32_t* nbr, bg_ctx_s* ctx, cudaStream_t st) {
    using Gm = Geo<K>;
    // points per chunk: the id buffer stays near 1 GiB unless the caller
    // passed nbr_out, which then holds all ids
    int64_t per = q.m;
    if (!nbr) per = std::min<int64_t>(q.m, std::max<int64_t>(4096, ((int64_t)1 << 28) / k));
    const size_t flag_bytes = 256;
    const size_t id_bytes = nbr ? 0 : (size_t)per * k * sizeof(int32_t);
    void* scratch = nullptr;
    const bool flagged = !query_by_lanes<K>(per);
    const size_t bytes = id_bytes + (flagged ? flag_bytes : 0);
    bg_status rc = bytes ? dalloc(ctx, &scratch, bytes, st) : BG_OK;
    if (rc != BG_OK) return rc;
    int* flag = flagged ? (int*)((char*)scratch + id_bytes) : nullptr;
    const cudaError_t ea = cudaFuncSetAttribute(
        k_okrige_solve_pts<K, kSph>, cudaFuncAttributeMaxDynamicSharedMemorySize, Gm::SMEM);
    if (ea != cudaSuccess) {
        if (scratch) dfree(ctx, scratch, bytes, st);
        return cuda_fail(ea, "solve shared-memory size");
    }
    for (int64_t p0 = 0; p0 < q.m; p0 += per) {
        const int64_t p1 = std::min<int64_t>(q.m, p0 + per);
        const int64_t n = p1 - p0;
        int32_t* chunk_ids = nbr ? nbr + p0 * k : (int32_t*)scratch;
        const int64_t stride = nbr ? 0 : n;
        cudaError_t e = flag ? cudaMemsetAsync(flag, 0, sizeof(int), st) : cudaSuccess;
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "memset");
            break;
        }
        const int len = strip_len_for(n);
        const int64_t nb = ((n + len - 1) / len + 127) / 128;
        {
            ProfScope ps(ctx, kProfKnnIds, n, st);
            if (query_by_lanes<K>(n))
                k_knn_ids_query<query_lanes(K)><<<query_blocks<K>(n), 32 * kQueryWarps, 0, st>>>(
                    h, q, p0, n, k, chunk_ids, stride, flag);
            else if (len == 1)
                k_knn_ids_pts<K, 1><<<(unsigned)nb, 128, 0, st>>>(h, q, k, p0, p1, chunk_ids, stride, flag);
            else if (len == 2)
                k_knn_ids_pts<K, 2><<<(unsigned)nb, 128, 0, st>>>(h, q, k, p0, p1, chunk_ids, stride, flag);
            else
                k_knn_ids_pts<K, 4><<<(unsigned)nb, 128, 0, st>>>(h, q, k, p0, p1, chunk_ids, stride, flag);
        }
        k_knn_ids_pts_wide<K><<<(unsigned)std::min<int64_t>((n + 127) / 128, 152 * 4), 128, 0, st>>>(
            h, q, k, p0, p1, chunk_ids, stride, flag);
        const int64_t batches = (n + kSolveSystems - 1) / kSolveSystems;
        const int bper = solve_batches_per_block<K>(batches);
        {
            ProfScope ps(ctx, kProfSolve, n, st);
            k_okrige_solve_pts<K, kSph>
                <<<(unsigned)((batches + bper - 1) / bper), Gm::THREADS, Gm::SMEM, st>>>(
                    h, q, k, p, p0, n, IdsView{chunk_ids, stride, 0, 0, 0}, depth, var, bper);
        }
        note_launches(3);
        e = cudaGetLastError();
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "kriging launch");
            break;
        }
    }
    if (scratch) dfree(ctx, scratch, bytes, st);
    return rc;
}

}  // namespace

bg_status launch_okrige_points(const bg_soundings_s* s, const PointsView& q, int k,
                               const OkParams& p, float* depth, float* var, int32_t* nbr,
                               cudaStream_t st) {
    if (q.m == 0) return BG_OK;
    HashView h = s->h;
    const int K = k <= 4 ? 4 : k <= 8 ? 8 : k <= 16 ? 16 : 32;
    h.r0 = start_halfwidth(s, K);
    const bool sph = p.model == BG_VARIOGRAM_SPHERICAL;
#define BG_OK_CASE(KK) \
    (sph ? launch_pts_k<KK, true>(h, q, k, p, depth, var, nbr, s->ctx, st) \
         : launch_pts_k<KK, false>(h, q, k, p, depth, var, nbr, s->ctx, st))
    switch (K) {
        case 4: return BG_OK_CASE(4);
        case 8: return BG_OK_CASE(8);
        case 16: return BG_OK_CASE(16);
        default: return BG_OK_CASE(32);
    }
#undef BG_OK_CASE
}

bg_status launch_okrige(const bg_soundings_s* s, const GridView& g, int k, const OkParams& p,
                        float* depth, float* var, int32_t* nbr, cudaStream_t st,
                        const IdwFuse* fz, const HostOut* ho) {
    HashView h = s->h;
    const int K = k <= 4 ? 4 : k <= 8 ? 8 : k <= 16 ? 16 : 32;
    if (fz && K != 32) {
        // the fused kernel is built for the largest system only: the IDW takes its
        // own pass (the same depths: idw_from sums in the same fixed order)
        bg_status rc = launch_idw(s, g, fz->k, fz->power, fz->out, nullptr, st);
        if (rc != BG_OK) return rc;
        if (ho && ho->idw) {  // the whole IDW grid is done: copy it now
            HostOut only_idw = *ho;
            only_idw.depth = only_idw.var = nullptr;
            rc = copy_rows_to_host(&only_idw, 0, (int64_t)g.nx * g.ny, fz->out, nullptr, nullptr, st);
            if (rc != BG_OK) return rc;
        }
        fz = nullptr;
    }
    h.r0 = start_halfwidth(s, K);
    const bool sph = p.model == BG_VARIOGRAM_SPHERICAL;
#define BG_OK_CASE(KK) \
    (sph ? launch_k<KK, true>(s, h, g, k, p, depth, var, nbr, s->ctx, st, fz, ho) \
         : launch_k<KK, false>(s, h, g, k, p, depth, var, nbr, s->ctx, st, fz, ho))
    switch (K) {
        case 4: return BG_OK_CASE(4);
        case 8: return BG_OK_CASE(8);
        case 16: return BG_OK_CASE(16);
        default: return BG_OK_CASE(32);
    }
#undef BG_OK_CASE
}

}  // namespace bg
