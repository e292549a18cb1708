// rt_trace.cu -- visibility of a ray set (Eq. 13-15, Sec. 4.1-4.2).
//
// One persistent launch: each warp (or group of lanes) repeatedly takes a work
// item from a device counter.  For a full implicit set (every Gaussian x K
// directions) an item is a shaft group x one direction (strategy 3), a ray slot
// (lane refill, lane groups) or 32 Gaussians adjacent in Morton order x one
// direction (the other packets and walks), so that a warp's rays start close
// together and, in a direction set, are parallel.  Items are ordered in
// sweeps: `order_block` tiles or groups for direction 0, the same for direction
// 1, ... .  The default, one per sweep, hands out its K directions in turn: the
// rows T[g, 0..K) are written within a short window (whole sectors merge in L2)
// and the warps in flight start in the same region of the tree (packets:
// sweeps of 64 to 62,500 tiles measured 0.6-2 % slower on the 2M-Gaussian object
// scene; lane refill: no difference from 1 to 4,096).  Explicit ray lists and id
// subsets are taken in the given order.
#include <string.h>

#include <algorithm>

#include "rt_shaft.cuh"

namespace {

// Resident blocks per SM the trace kernels are compiled for (register cap).
constexpr int kTraceBlocks = 8;

// Packets of rays with directions of their own take 60 registers where they are
// let, which costs the ninth block and 2 to 3 %.
template <int STRAT, bool COUNT>
__global__ void __launch_bounds__(128, STRAT == 5 ? kRefillBlocks : STRAT == 2 && !COUNT ? 9 : kTraceBlocks)
    k_trace(BvhDev b, RaySetDev rs, TraceJob job, float *T_out, TraceAux aux, unsigned long long *work) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    constexpr bool packet = STRAT == 2 || STRAT == 3;
    __shared__ int2 stk_all[packet ? 4 * RT_WIDE_STACK : 1];
    int2 *stk = stk_all + (packet ? (threadIdx.x >> 5) * RT_WIDE_STACK : 0);
    WorkCounts wc = {0, 0, 0};
    unsigned long long rays_done = 0;
    if constexpr (STRAT == 5) {  // per-ray slots with lane refill (full implicit sets)
        trace_refill<COUNT>(b, rs, job, T_out, aux, work, wc, rays_done);
        flush_counts<COUNT>(aux, wc, rays_done);
        return;
    }
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(work, 1ull);
        item = __shfl_sync(FULL, item, 0);
        if ((int64_t)item >= job.n_items) break;
        int64_t n_out = job.n_out;
        if (job.dyn_count) {
            const int64_t c = (int64_t)*job.dyn_count;
            n_out = c < n_out ? c : n_out;
            if ((int64_t)item * 32 >= n_out) break;
        }
        trace_item<STRAT, COUNT>(b, rs, job, T_out, aux, (int64_t)item, n_out, wc, rays_done, stk);
    }
    flush_counts<COUNT>(aux, wc, rays_done);
}

// Strategy 6: a group of lanes per ray.
template <int LANES, bool COUNT>
__global__ void __launch_bounds__(128, kTraceBlocks) k_trace_lanes(BvhDev b, RaySetDev rs, TraceJob job,
                                                                          float *T_out, TraceAux aux,
                                                                          unsigned long long *work) {
    __shared__ uint32_t stk[128 * kLaneStack<LANES>];
    __shared__ int32_t queue[kLeafQueue * 128];
    WorkCounts wc = {0, 0, 0};
    unsigned long long rays_done = 0;
    trace_lane_group<LANES, COUNT>(b, rs, job, T_out, aux, work, stk + threadIdx.x / LANES * (LANES * kLaneStack<LANES>),
                                   queue + threadIdx.x, wc, rays_done);
    flush_counts<COUNT>(aux, wc, rays_done);
}

// Strategy 3 of a direction set: an item is a shaft group and a direction.
__global__ void __launch_bounds__(128, kShaftBlocks) k_trace_shaft(BvhDev b, RaySetDev rs, TraceJob job,
                                                                          float *T_out, int *status,
                                                                          unsigned long long *work) {
    __shared__ ShaftSmem<false> sm[4];
    for (;;) {
        unsigned long long item = 0;
        if ((threadIdx.x & 31) == 0) item = atomicAdd(work, 1ull);
        item = __shfl_sync(0xffffffffu, item, 0);
        if ((int64_t)item >= job.n_items) break;
        shaft_item(b, rs, job, T_out, (int64_t)item, status, sm[threadIdx.x >> 5]);
    }
}

// Sort keys of an id list (per-ray traversal of long lists): rays of one
// direction index in the tree's (Morton) order of their Gaussians, so that
// neighbouring threads walk neighbouring parts of the tree.  DIRS: key =
// k * n + sorted position; hemisphere and env-map sets (directions differ
// per Gaussian or per sample): the sorted position alone.  Invalid ids sort
// last and are reported by the trace.
__global__ void k_list_keys(BvhDev b, RaySetDev rs, int64_t m, uint32_t *keys, int32_t *vals) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t rid = rs.ray_ids[i];
        uint32_t key = 0xffffffffu;
        if (rid >= 0 && rid < rs.n_rays) {
            const int64_t g = rid / rs.K;
            const uint32_t p = (uint32_t)b.rank[g];
            key = rs.kind == RT_RAYS_DIRS ? (uint32_t)(rid - g * rs.K) * (uint32_t)b.n + p : p;
        }
        keys[i] = key;
        vals[i] = (int32_t)i;
    }
}
// The list in sorted order and each entry's place in the caller's list.
__global__ void k_list_perm(const int64_t *ids, const int32_t *vals, int64_t m, int64_t *sorted_ids,
                            int64_t *out_index) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t i = vals[j];
        sorted_ids[j] = ids[i];
        out_index[j] = i;
    }
}

int persistent_blocks(const void *kernel, int threads) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    return per_sm * rt_num_sms();
}

// Lanes per ray that AUTO takes for m rays.  300k object scene, shadow rays in
// no order, us with 32 / 16 / 8 / 4 lanes: 2,000 rays 50 / 69 / 101 / 176; 20,000
// 122 / 122 / 154 / 230; 100,000 433 / 368 / 325 / 361; 250,000 1,019 / 836 / 683 /
// 667; 600,000 2,384 / 1,929 / 1,491 / 1,322.  Beyond 2^20 Gaussians nodes and records exceed the L2
// cache and more lanes hide its misses: 1M rays of the 2M scene 6,138 / 5,724 /
// 5,302 / 6,443.  4 lanes' stack holds a walk of single nodes through 36 levels.
// RT_KERNEL_WARP_RAY asked for by name, and the surrogate's fallback with it, keep
// 32 whatever the number: the order of a ray's factors follows the lanes, and T
// of these is to be the same bit for bit in a full set and in any list.  (A
// fallback list's length is also only known on the device: lanes by its bound took
// 113 us for the 2,900 of 70,000 rays that fall back on the 200k scene, 32
// lanes 74; for 134,000 of 2M rays, the other way, 820 and 976.)
int lanes_for(int64_t m, const BvhDev &b) {
    if (m <= 8192) return 32;
    if (m <= 65536) return 16;
    return m <= 262144 || b.levels > 36 || b.n > (int64_t(1) << 20) ? 8 : 4;
}

// A full set traced by groups of lanes.  Hemisphere and environment sets, us,
// lanes against one thread per ray or lane refill, whichever is less, by the rays
// per shaft group (how dense the scene is):
//   uniform 1k: x 16 30 / 66 and 36 / 67; 2k (5): x 32 96 / 138 and 113 / 139
//   uniform 10 to 28: 4k x 16 122 / 204 and 141 / 211, x 32 205 / 262 and 244 / 268;
//     20k x 16 (320k rays) 870 / 1,095 and 1,001 / 1,108, x 32 1,625 / 1,690 and
//     1,897 / 1,725; 60k x 8 (480k) 1,695 / 1,860 and 1,912 / 1,882
//   object 2 (4k): x 8 57 / 70 and 67 / 72, x 12 78 / 86 and 91 / 78, x 16 99 / 83
//     and 117 / 83
//   object 8 (20k): x 8 200 / 242 and 266 / 274, x 16 338 / 330 and 438 / 378, x 32
//     627 / 471 and 827 / 552
//   object 11 to 24: 60k x 4 (240k rays) 461 / 490 and 572 / 552, x 8 704 / 670 and
//     913 / 770; 400k x 2 1,982 / 2,110
// A lane group works out a ray's direction in every lane, which environment
// samples make long.  Direction sets against shaft packets or one thread per ray:
// uniform 3k x 8 52 / 80, x 32 118 / 103; 30k x 1 144 / 247, x 4 398 / 258; object
// 4k x 8 55 / 90, x 16 94 / 85; 500 x 16 26 / 26, x 64 42 / 28.
bool small_set_takes_lanes(const rt_bvh *bvh, int32_t kind, int32_t K, int64_t rays) {
    if (kind == RT_RAYS_DIRS) return rays <= (int64_t(1) << 15) && K <= 16;
    const bool dense = bvh->n >= 9 * bvh->n_groups, denser = bvh->n >= 16 * bvh->n_groups;
    if (rays > (int64_t(1) << (K <= 2 ? 20 : denser ? 19 : 18))) return false;
    if (K <= 8 || dense) return K <= 32;
    if (K <= 16 && (kind == RT_RAYS_HEMI || rays <= (int64_t(1) << 14))) return true;
    return K <= 32 && rt_shaft_pays(bvh) && rays <= (int64_t(1) << 17);
}

// No more blocks than the rays need, and with 32 lanes, for few rays, the nodes
// kept in L1: 1,000 to 2,000 rays of scenes of 500 to 4,000 Gaussians, bound by
// the launch and one ray's walk, 14.9 to 20.6 us without either, 13.4 to 18.6 with.
template <bool COUNT>
void launch_lanes(int lanes, const BvhDev &b, const RaySetDev &rs, const TraceJob &job, float *T_out,
                  const TraceAux &aux, cudaStream_t st, unsigned long long *work) {
#define RT_LANES(L)                                                                                      \
    k_trace_lanes<L, COUNT><<<(int)std::min<int64_t>((job.n_out * L + 127) / 128,                         \
                                                     persistent_blocks((const void *)k_trace_lanes<L, COUNT>, 128)), \
                              128, 0, st>>>(b, rs, job, T_out, aux, work)
    switch (lanes) {
        case 32: RT_LANES(32); break;
        case 16: RT_LANES(16); break;
        case 8: RT_LANES(8); break;
        default: RT_LANES(4);
    }
#undef RT_LANES
}

}  // namespace

// Launch the single-scene kernel of strategy 0 to 5 on an explicit job (used by
// the autotuner).
rt_status rt_trace_launch_job(const BvhDev &b, const RaySetDev &rs, const TraceJob &job, float *T_out,
                              int strat, rt_stream_t stream, unsigned long long *work) {
    TraceAux aux;
    memset(&aux, 0, sizeof(aux));
    aux.status = rt_status_ptr();
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(work, 0, sizeof(unsigned long long), st) != cudaSuccess) return RT_ERR_CUDA;
    const int threads = 128;
    if (strat == 5 && b.wide && job.mode == MODE_FULL) {
        int grid = persistent_blocks((const void *)k_trace<5, false>, threads);
        k_trace<5, false><<<grid, threads, 0, st>>>(b, rs, job, T_out, aux, work);
    } else if (strat >= 4 && b.wide) {
        int grid = persistent_blocks((const void *)k_trace<4, false>, threads);
        k_trace<4, false><<<grid, threads, 0, st>>>(b, rs, job, T_out, aux, work);
    } else if (strat >= 4) {
        int grid = persistent_blocks((const void *)k_trace<0, false>, threads);
        k_trace<0, false><<<grid, threads, 0, st>>>(b, rs, job, T_out, aux, work);
    } else if (strat >= 2 && b.wide) {
        if (job.mode == MODE_FULL && rs.kind == RT_RAYS_DIRS) {
            int grid = persistent_blocks((const void *)k_trace_shaft, threads);
            k_trace_shaft<<<grid, threads, 0, st>>>(b, rs, job, T_out, aux.status, work);
        } else {
            int grid = persistent_blocks((const void *)k_trace<2, false>, threads);
            k_trace<2, false><<<grid, threads, 0, st>>>(b, rs, job, T_out, aux, work);
        }
    } else if (strat >= 1) {
        int grid = persistent_blocks((const void *)k_trace<1, false>, threads);
        k_trace<1, false><<<grid, threads, 0, st>>>(b, rs, job, T_out, aux, work);
    } else {
        int grid = persistent_blocks((const void *)k_trace<0, false>, threads);
        k_trace<0, false><<<grid, threads, 0, st>>>(b, rs, job, T_out, aux, work);
    }
    return rt_check_launch();
}

// Shared by rt_trace_visibility and the batched launch.
rt_status rt_trace_launch(const rt_bvh *bvh, const rt_rayspec *rays, float *T_out,
                          const rt_trace_opts *opts, rt_stream_t stream, unsigned long long *work) {
    RaySetDev rs;
    int64_t count = 0;
    RT_TRY(rt_rayset_dev(bvh, rays, &rs, &count));
    if (count > 0 && !T_out) return RT_ERR_INVALID_ARG;
    rt_trace_opts o;
    memset(&o, 0, sizeof(o));
    if (opts) o = *opts;
    if (o.kernel < 0 || o.kernel > 6 || o.order_block < 0 || o.block_threads < 0) return RT_ERR_INVALID_ARG;
    if ((o.hit_ids && (o.hit_cap <= 0 || !o.hit_count)) ) return RT_ERR_INVALID_ARG;
    if (count == 0) return RT_OK;

    TraceJob job;
    job.out_index = nullptr;
    job.dyn_count = nullptr;
    job.n_out = count;
    job.order_block = 1;
    job.n_tiles = 0;
    job.tile_base = 0;
    if (rays->kind == RT_RAYS_EXPLICIT) job.mode = MODE_EXPLICIT;
    else if (rays->ray_ids) job.mode = MODE_IDS;
    else job.mode = MODE_FULL;
    if (job.mode == MODE_FULL) {
        job.n_tiles = (bvh->n + 31) / 32;
        int64_t B = o.order_block > 0 ? o.order_block : 1;
        if (B > job.n_tiles) B = job.n_tiles;
        job.order_block = (int32_t)B;
        job.n_items = job.n_tiles * rs.K;
    } else {
        job.n_items = (count + 31) / 32;
    }
    int strat = o.kernel == RT_KERNEL_WARP_RAY ? 6 : o.kernel == RT_KERNEL_RAY_REFILL ? 5
              : o.kernel == RT_KERNEL_RAY_WIDE ? 4 : o.kernel == RT_KERNEL_WIDE ? 2
              : o.kernel == RT_KERNEL_PACKET ? 1 : 0;
    // AUTO:
    // - a small full set: a group of lanes per ray (lanes_for), which is bound
    //   by one ray's latency less than the others (small_set_takes_lanes);
    // - a direction set: shaft packets where the groups are large enough
    //   (rt_shaft_pays), else one thread per ray, farthest child first, as with
    //   counters or a hit log, which shaft packets do not keep (2M object scene x
    //   8, counted 96 ms, packets 102; 600k x 16 31 / 36);
    // - env-map and hemisphere sets (directions differ across a tile): the
    //   per-ray walk with lane refill, up to 2^18 rays (2^17 in dense scenes)
    //   one thread per ray, whose latency is lower (environment sets, us, thread /
    //   refill: object 4k x 32 102 / 125, x 64 143 / 157, 20k x 16 428 / 378; uniform
    //   4k x 32 280 / 268, x 64 418 / 329);
    // - explicit rays and id lists (scattered rays): a group of lanes per ray
    //   up to 2^22 rays (lanes_for; one thread per ray takes 570 us for 2,000
    //   rays of the 300k scene, 2.4 ms for 600,000), and one thread per ray
    //   over the 4-wide tree for longer lists, which are sorted.
    const int64_t thread_max = int64_t(1) << (bvh->n >= 9 * bvh->n_groups ? 17 : 18);
    if (o.kernel == RT_KERNEL_AUTO && job.mode == MODE_FULL)
        strat = !o.counters && !o.hit_ids && small_set_takes_lanes(bvh, rays->kind, rs.K, count) ? 6
                : rays->kind != RT_RAYS_DIRS ? (count <= thread_max ? 4 : 5)
                : !o.counters && !o.hit_ids && rt_shaft_pays(bvh) ? 2
                                                                  : 4;
    if (o.kernel == RT_KERNEL_AUTO && job.mode != MODE_FULL) strat = count <= (int64_t(1) << 22) ? 6 : 4;
    // lanes per ray keep no hit log
    if (strat == 6 && o.hit_ids) strat = 4;
    // lane refill needs the 4-wide tree and a full implicit set, and keeps no hit log
    if (strat == 5 && (bvh->n_wide == 0 || job.mode != MODE_FULL || o.hit_ids)) strat = 4;
    if (strat == 2 && bvh->n_wide == 0) strat = 1;
    if ((strat == 4 || strat == 6) && bvh->n_wide == 0) strat = 0;  // fewer than two Gaussians
    // a shared direction: shaft packets, which count no single ray's tests and
    // keep no hit log (then the plain packet walk)
    const bool shared_dir = job.mode == MODE_FULL && rays->kind == RT_RAYS_DIRS;
    if (strat == 2 && shared_dir && !o.counters && !o.hit_ids) strat = 3;

    TraceAux aux;
    aux.counters = (unsigned long long *)o.counters;
    aux.hit_ids = o.hit_ids;
    aux.hit_count = o.hit_count;
    aux.cap = o.hit_cap;
    aux.status = rt_status_ptr();
    BvhDev b = bvh_dev(bvh);
    cudaStream_t st = (cudaStream_t)stream;

    // AUTO on a long id list (per-ray traversal): trace it in the order of
    // (direction, the tree's order of the Gaussians), each T written back to
    // its place in the caller's list (2M object scene, 64M stratified
    // held-out rays: 141 against 111 M rays/s); each ray's traversal, and so
    // its T, is the same in any order
    void *sort_blk = nullptr;
    if (o.kernel == RT_KERNEL_AUTO && job.mode == MODE_IDS && strat == 4 && count < (int64_t(1) << 31) &&
        (uint64_t)rs.K * (uint64_t)bvh->n < (uint64_t(1) << 32)) {
        auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
        const size_t b4 = up(size_t(count) * 4), b8 = up(size_t(count) * 8);
        RT_TRY(rt_alloc(&sort_blk, 2 * b4 + 2 * b8, stream));
        uint32_t *keys = (uint32_t *)sort_blk;
        int32_t *vals = (int32_t *)((char *)sort_blk + b4);
        int64_t *sids = (int64_t *)((char *)sort_blk + 2 * b4), *oidx = (int64_t *)((char *)sort_blk + 2 * b4 + b8);
        const int g = rt_num_sms() * 8;
        k_list_keys<<<g, 256, 0, (cudaStream_t)stream>>>(bvh_dev(bvh), rs, count, keys, vals);
        rt_status r = rt_check_launch();
        if (r == RT_OK) r = rt_sort_pairs_u32(keys, vals, count, 32, stream);
        if (r == RT_OK) {
            k_list_perm<<<g, 256, 0, (cudaStream_t)stream>>>(rs.ray_ids, vals, count, sids, oidx);
            r = rt_check_launch();
        }
        if (r != RT_OK) {
            rt_free(sort_blk, stream);
            return r;
        }
        rs.ray_ids = sids;
        job.out_index = oidx;
    }
    bool own = false;
    if (!work) {
        if (rt_alloc((void **)&work, sizeof(unsigned long long), stream) != RT_OK) {
            if (sort_blk) rt_free(sort_blk, stream);
            return RT_ERR_OOM;
        }
        own = true;
    }
    rt_status res = RT_OK;
    if (cudaMemsetAsync(work, 0, sizeof(unsigned long long), st) != cudaSuccess) res = RT_ERR_CUDA;
    // counts without a log: none is kept, and the walks that keep no log write none
    if (o.hit_count && !o.hit_ids && (strat == 3 || strat >= 5) &&
        cudaMemsetAsync(o.hit_count, 0, sizeof(int32_t) * (size_t)count, st) != cudaSuccess)
        res = RT_ERR_CUDA;
    if (res == RT_OK) {
        const int threads = 128;
        const bool count = aux.counters != nullptr;
#define RT_LAUNCH(S, C)                                                                     \
    do {                                                                                    \
        int grid = persistent_blocks((const void *)k_trace<S, C>, threads);                 \
        k_trace<S, C><<<grid, threads, 0, st>>>(b, rs, job, T_out, aux, work);              \
    } while (0)
        if (strat == 6) {
            const int lanes = o.kernel == RT_KERNEL_WARP_RAY ? 32 : lanes_for(job.n_out, b);
            if (count) launch_lanes<true>(lanes, b, rs, job, T_out, aux, st, work);
            else launch_lanes<false>(lanes, b, rs, job, T_out, aux, st, work);
        }
        else if (strat == 5) { if (count) RT_LAUNCH(5, true); else RT_LAUNCH(5, false); }
        else if (strat == 4) { if (count) RT_LAUNCH(4, true); else RT_LAUNCH(4, false); }
        else if (strat == 3) {
            // its items are shaft groups instead of tiles
            job.n_tiles = bvh->n_groups;
            if (job.order_block > job.n_tiles) job.order_block = (int32_t)job.n_tiles;
            job.n_items = job.n_tiles * rs.K;
            int grid = persistent_blocks((const void *)k_trace_shaft, threads);
            k_trace_shaft<<<grid, threads, 0, st>>>(b, rs, job, T_out, aux.status, work);
        }
        else if (strat == 2 && shared_dir) { if (count) RT_LAUNCH(3, true); else RT_LAUNCH(3, false); }
        else if (strat == 2) { if (count) RT_LAUNCH(2, true); else RT_LAUNCH(2, false); }
        else if (strat == 1) { if (count) RT_LAUNCH(1, true); else RT_LAUNCH(1, false); }
        else { if (count) RT_LAUNCH(0, true); else RT_LAUNCH(0, false); }
#undef RT_LAUNCH
        res = rt_check_launch();
    }
    if (own) rt_free(work, stream);
    if (sort_blk) rt_free(sort_blk, stream);
    return res;
}

// Trace the rays listed in ray_ids[0 .. *count) (device count, at most
// max_count) of an implicit set and write T_out[out_index[i]].
rt_status rt_trace_launch_list(const rt_bvh *bvh, const rt_rayspec *rays, const int64_t *ray_ids,
                               const int64_t *out_index, const unsigned long long *count, int64_t max_count,
                               float *T_out, rt_stream_t stream, unsigned long long *work) {
    if (rays->kind == RT_RAYS_EXPLICIT || !ray_ids || !out_index || !count || !work) return RT_ERR_INVALID_ARG;
    RaySetDev rs;
    int64_t c = 0;
    rt_rayspec tmp = *rays;
    tmp.ray_ids = nullptr;
    RT_TRY(rt_rayset_dev(bvh, &tmp, &rs, &c));
    rs.ray_ids = ray_ids;
    if (max_count <= 0) return RT_OK;
    TraceJob job;
    job.mode = MODE_IDS;
    job.out_index = out_index;
    job.dyn_count = count;
    job.n_out = max_count;
    job.n_tiles = 0;
    job.tile_base = 0;
    job.order_block = 1;
    job.n_items = (max_count + 31) / 32;
    TraceAux aux;
    memset(&aux, 0, sizeof(aux));
    aux.status = rt_status_ptr();
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(work, 0, sizeof(unsigned long long), st) != cudaSuccess) return RT_ERR_CUDA;
    const int threads = 128;
    // the listed rays are few and scattered: RT_KERNEL_WARP_RAY
    const BvhDev b = bvh_dev(bvh);
    if (bvh->n_wide > 0) {
        launch_lanes<false>(32, b, rs, job, T_out, aux, st, work);
    } else {
        int grid = persistent_blocks((const void *)k_trace<0, false>, threads);
        k_trace<0, false><<<grid, threads, 0, st>>>(b, rs, job, T_out, aux, work);
    }
    return rt_check_launch();
}

extern "C" rt_status rt_trace_visibility(const rt_bvh *bvh, const rt_rayspec *rays, float *T_out,
                                         const rt_trace_opts *opts, rt_stream_t stream) {
    if (!bvh || !rays) return RT_ERR_INVALID_ARG;
    return rt_trace_launch(bvh, rays, T_out, opts, stream, nullptr);
}

extern "C" rt_status rt_trace_visibility_dirs(const rt_bvh *bvh, const float *dirs, int32_t k,
                                              float *T_out, const rt_trace_opts *opts,
                                              rt_stream_t stream) {
    if (!bvh) return RT_ERR_INVALID_ARG;
    rt_rayspec rs;
    memset(&rs, 0, sizeof(rs));
    rs.kind = RT_RAYS_DIRS;
    rs.n_dirs = k;
    rs.dirs = dirs;
    return rt_trace_launch(bvh, &rs, T_out, opts, stream, nullptr);
}

// ---------------------------------------------------------------------------
// The precompute from host buffers: copies in, build, trace, copy out, all on
// one stream.
// ---------------------------------------------------------------------------
extern "C" rt_status rt_visibility_dirs_host(const float *mean, const float *scale, const float *quat,
                                             const float *opacity, int64_t n, const float *dirs, int32_t k,
                                             const rt_params *params, const rt_trace_opts *opts, float *T_host,
                                             rt_stream_t stream) {
    if (n < 0 || k < 0 || n >= (int64_t(1) << 31)) return RT_ERR_INVALID_ARG;
    const int64_t R = n * (int64_t)k;
    if (R == 0) return RT_OK;
    if (R >= (int64_t(1) << 40) || !mean || !scale || !quat || !opacity || !dirs || !T_host)
        return RT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t b3 = up(size_t(n) * 12), b4 = up(size_t(n) * 16), b1 = up(size_t(n) * 4), bd = up(size_t(k) * 12);
    void *blk = nullptr;
    rt_status s = rt_alloc(&blk, 2 * b3 + b4 + b1 + bd, stream);
    if (s != RT_OK) return s;
    char *base = (char *)blk;
    float *d_mean = (float *)base, *d_scale = (float *)(base + b3), *d_quat = (float *)(base + 2 * b3),
          *d_opac = (float *)(base + 2 * b3 + b4), *d_dirs = (float *)(base + 2 * b3 + b4 + b1);
    const struct { void *dst; const void *src; size_t bytes; } in[5] = {
        {d_mean, mean, size_t(n) * 12}, {d_scale, scale, size_t(n) * 12}, {d_quat, quat, size_t(n) * 16},
        {d_opac, opacity, size_t(n) * 4}, {d_dirs, dirs, size_t(k) * 12}};
    for (const auto &c : in) {
        if (cudaMemcpyAsync(c.dst, c.src, c.bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) {
            cudaGetLastError();
            rt_free(blk, stream);
            return RT_ERR_CUDA;
        }
    }
    rt_bvh *bvh = nullptr;
    s = rt_build_bvh(d_mean, d_scale, d_quat, d_opac, n, params, stream, &bvh);
    if (s != RT_OK) {
        rt_free(blk, stream);
        return s;
    }
    float *d_T = nullptr;
    s = rt_alloc((void **)&d_T, size_t(R) * 4, stream);
    if (s == RT_OK) {
        s = rt_trace_visibility_dirs(bvh, d_dirs, k, d_T, opts, stream);
        if (s == RT_OK && cudaMemcpyAsync(T_host, d_T, size_t(R) * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) {
            cudaGetLastError();
            s = RT_ERR_CUDA;
        }
        rt_free(d_T, stream);
    }
    rt_bvh_destroy(bvh, stream);
    rt_free(blk, stream);
    return s;
}

// ---------------------------------------------------------------------------
// Materialised rays of an implicit set (for inspection and the adjoint)
// ---------------------------------------------------------------------------
namespace {
__global__ void k_materialize(BvhDev b, RaySetDev rs, const int64_t *ids, int64_t m, float *ro,
                              float *rd, int32_t *rsrc, int *status) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        int64_t rid = ids[i];
        if (rid < 0 || rid >= rs.n_rays) {
            rt_set_error(status, RT_ERR_INVALID_ARG);
            continue;
        }
        int64_t g = rid / rs.K;
        int32_t k = (int32_t)(rid - g * rs.K);
        int32_t p = b.rank[g];
        float3 o, d;
        implicit_ray(rs, rid, k, g, __ldg(b.gauss + 4 * (int64_t)p), o, d);
        ro[3 * i] = o.x; ro[3 * i + 1] = o.y; ro[3 * i + 2] = o.z;
        rd[3 * i] = d.x; rd[3 * i + 1] = d.y; rd[3 * i + 2] = d.z;
        if (rsrc) rsrc[i] = (int32_t)g;
    }
}
}  // namespace

extern "C" rt_status rt_materialize_rays(const rt_bvh *bvh, const rt_rayspec *rays,
                                         const int64_t *ray_ids, int64_t m, float *ray_o,
                                         float *ray_d, int32_t *ray_src, rt_stream_t stream) {
    if (!bvh || !rays || m < 0) return RT_ERR_INVALID_ARG;
    if (rays->kind == RT_RAYS_EXPLICIT) return RT_ERR_INVALID_ARG;
    if (m == 0) return RT_OK;
    if (!ray_ids || !ray_o || !ray_d) return RT_ERR_INVALID_ARG;
    RaySetDev rs;
    int64_t c;
    rt_rayspec tmp = *rays;
    tmp.ray_ids = nullptr;
    RT_TRY(rt_rayset_dev(bvh, &tmp, &rs, &c));
    int grid = (int)((m + 255) / 256);
    if (grid > rt_num_sms() * 8) grid = rt_num_sms() * 8;
    k_materialize<<<grid, 256, 0, (cudaStream_t)stream>>>(bvh_dev(bvh), rs, ray_ids, m, ray_o, ray_d,
                                                          ray_src, rt_status_ptr());
    return rt_check_launch();
}
