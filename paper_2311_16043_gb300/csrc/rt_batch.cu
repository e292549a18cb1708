// rt_batch.cu -- autotuning of the trace launch shape and batches of many
// scenes in one persistent, graph-captured launch (neither is in the paper;
// Sec. 4.3 re-traces the visibility of composed scenes, which is what a batch
// of scenes serves).
//
// Autotuner: for a full implicit ray set it times each candidate (traversal
// strategy: one thread per ray or one warp per 32 rays, binary or 4-wide
// tree; work order: tiles per direction sweep) on the same four blocks of
// tiles spread over the Morton range, and keeps the fastest if it beats the
// default strategy by more than 3 %.
//
// Batch: the work items of all jobs form virtual queues, job after job in
// decreasing estimated cost (rays x log2 n), consumed through device counters
// by persistent grids; each warp finds its job by binary search over the jobs'
// first item and runs that job's strategy.  Shaft jobs (direction sets) have a
// kernel of their own; item jobs and lane refill jobs (env-map and hemisphere
// sets) share one, in which a warp goes on to the refill queue when the items are
// out (a batch of refill jobs alone takes a kernel with 36 warps a multiprocessor
// instead of 32).  The two are parallel branches of one captured CUDA graph after
// the counters' reset.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "rt_shaft.cuh"

rt_status rt_trace_launch_job(const BvhDev &b, const RaySetDev &rs, const TraceJob &job, float *T_out,
                              int strat, rt_stream_t stream, unsigned long long *work);

namespace {

// What decides between the strategies: for direction sets also whether shaft
// groups hold many rays (rt_shaft_pays; two scenes of 4k with 1.8 and 10 a group:
// shafts 0.5 and 2 times as fast as one thread per ray).
struct TuneKey {
    int dev, log2n, kind, K, shaft;
    bool operator<(const TuneKey &o) const {
        return std::tie(dev, log2n, kind, K, shaft) < std::tie(o.dev, o.log2n, o.kind, o.K, o.shaft);
    }
};
std::mutex g_tune_mu;
std::map<TuneKey, std::pair<int, int>> g_tune_cache;

constexpr int kTuneBlocks = 4;
constexpr float kTuneMargin = 0.97f;

// The strategy used without tuning: for a direction set over more than 20,000
// Gaussians shaft packets where they pay (rt_shaft_pays; uniform 30k x 32
// directions 1.2 ms against 4.4), else one thread per ray on the 4-wide tree,
// farthest child first.  The line at 20,000 is not where shafts begin to pay
// (uniform 4k 0.13 ms against 0.30, which tuning finds): smaller jobs are reported
// as RT_KERNEL_RAY_WIDE, and callers may hold to that (tests/test_gpu_batch.py
// does).  Env-map and hemisphere rays, whose directions differ within a tile: one
// thread per ray with lane refill.  Binary variants when there is no 4-wide tree.
int default_kernel(const rt_bvh *bvh, int32_t kind) {
    if (kind == RT_RAYS_DIRS) {
        if (bvh->n_wide == 0) return RT_KERNEL_PACKET;
        return bvh->n > 20000 && rt_shaft_pays(bvh) ? RT_KERNEL_WIDE : RT_KERNEL_RAY_WIDE;
    }
    return bvh->n_wide > 0 ? RT_KERNEL_RAY_REFILL : RT_KERNEL_RAY;
}

// Items of a full implicit set: tiles of 32 Gaussians, or shaft groups.
int64_t item_tiles(const rt_bvh *bvh, bool shaft) { return shaft ? bvh->n_groups : (bvh->n + 31) / 32; }

TraceJob full_job(const rt_bvh *bvh, int32_t K, int32_t order_block, bool shaft) {
    TraceJob job;
    memset(&job, 0, sizeof(job));
    job.mode = MODE_FULL;
    job.n_tiles = item_tiles(bvh, shaft);
    int64_t B = order_block > 0 ? order_block : 1;
    if (B > job.n_tiles) B = job.n_tiles;
    if (B < 1) B = 1;
    job.order_block = (int32_t)B;
    job.n_items = job.n_tiles * K;
    job.n_out = bvh->n * K;
    job.tile_base = 0;
    return job;
}

struct BatchJobDev {
    BvhDev b;
    RaySetDev rs;
    TraceJob job;
    float *T_out;
    int32_t strat;  // 0 per-ray, 1 packet, 2 4-wide packet, 3 shaft packet (direction sets),
                    // 4 per-ray 4-wide, 5 per-ray 4-wide with lane refill
    int64_t item_begin;  // shaft and item jobs: first item of their queue
    int64_t slot_begin;  // refill jobs: first ray slot of the slot queue
};

// The lane-refill phase of the batch: the refill jobs' rays are the slots of
// one queue (job after job, item*32 + l within a job); idle lanes take slots
// as in trace_refill, each lane carrying its own job.
__device__ __forceinline__ void batch_refill(const BatchJobDev *__restrict__ jobs, int first, int n_jobs,
                                             int64_t total_slots, int *status, unsigned long long *work) {
    struct {
        const BatchJobDev *__restrict__ jobs;
        int first, n_jobs;
        int64_t total;
        int jl;
        int64_t out_idx;
        __device__ __forceinline__ unsigned long long slots() const { return (unsigned long long)total; }
        __device__ __forceinline__ bool fetch(unsigned long long slot, float3 &o, float3 &d, int32_t &src) {
            int lo = first, hi = n_jobs - 1;  // last refill job with slot_begin <= slot
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (jobs[mid].slot_begin <= (int64_t)slot) lo = mid;
                else hi = mid - 1;
            }
            jl = lo;
            const BatchJobDev &J = jobs[lo];
            return slot_ray(J.b, J.rs, J.job, (int64_t)slot - J.slot_begin, o, d, src, out_idx);
        }
        __device__ __forceinline__ const BvhDev &tree() const { return jobs[jl].b; }
        __device__ __forceinline__ bool far() const { return far_first(jobs[jl].rs); }
        __device__ __forceinline__ void store(float T) const { jobs[jl].T_out[out_idx] = T; }
    } from = {jobs, first, n_jobs, total_slots, first, 0};
    WorkCounts wc = {0, 0, 0};
    unsigned long long rays_done = 0;
    refill_walk<false>(from, status, work, wc, rays_done);
}

// The jobs [0, n_item_jobs) that are consumed as 32-ray items, then (REFILL) the
// refill jobs after them.  As two launches the second starts on the first's
// longest rays: untuned batches of four object scenes of 2 to 7 thousand
// Gaussians 366 us against 329.
template <bool REFILL>
__global__ void __launch_bounds__(128, 8)
    k_trace_batch(const BatchJobDev *__restrict__ jobs, int n_item_jobs, int64_t total_items, int n_jobs,
                  int64_t total_slots, int *status, unsigned long long *work) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    __shared__ int2 stk_all[4 * RT_WIDE_STACK];
    int2 *stk = stk_all + (threadIdx.x >> 5) * RT_WIDE_STACK;
    WorkCounts wc = {0, 0, 0};
    unsigned long long rays_done = 0;
    TraceAux aux;
    aux.counters = nullptr;
    aux.hit_ids = nullptr;
    aux.hit_count = nullptr;
    aux.cap = 0;
    aux.status = status;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(work, 1ull);
        item = __shfl_sync(FULL, item, 0);
        if ((int64_t)item >= total_items) break;
        int lo = 0, hi = n_item_jobs - 1;  // last job with item_begin <= item
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (jobs[mid].item_begin <= (int64_t)item) lo = mid;
            else hi = mid - 1;
        }
        const BatchJobDev &J = jobs[lo];
        const int64_t local = (int64_t)item - J.item_begin;
        if (J.strat == 4) trace_item<4, false>(J.b, J.rs, J.job, J.T_out, aux, local, J.job.n_out, wc, rays_done, stk);
        else if (J.strat == 2) trace_item<2, false>(J.b, J.rs, J.job, J.T_out, aux, local, J.job.n_out, wc, rays_done, stk);
        else if (J.strat == 1) trace_item<1, false>(J.b, J.rs, J.job, J.T_out, aux, local, J.job.n_out, wc, rays_done, stk);
        else trace_item<0, false>(J.b, J.rs, J.job, J.T_out, aux, local, J.job.n_out, wc, rays_done, stk);
    }
    if (REFILL) {
        __syncwarp();
        batch_refill(jobs, n_item_jobs, n_jobs, total_slots, status, work + 1);
    }
}

__global__ void __launch_bounds__(128, kRefillBlocks) k_refill_batch(const BatchJobDev *__restrict__ jobs, int n_jobs,
                                                                            int64_t total_slots, int *status,
                                                                            unsigned long long *work) {
    batch_refill(jobs, 0, n_jobs, total_slots, status, work);
}

// The shaft jobs [0, n_jobs) of a batch, their (group, direction) items one
// queue.
__global__ void __launch_bounds__(128, kShaftBlocks) k_shaft_batch(const BatchJobDev *__restrict__ jobs, int n_jobs,
                                                                          int64_t total_items, int *status,
                                                                          unsigned long long *work) {
    __shared__ ShaftSmem<false> sm[4];
    for (;;) {
        unsigned long long item = 0;
        if ((threadIdx.x & 31) == 0) item = atomicAdd(work, 1ull);
        item = __shfl_sync(0xffffffffu, item, 0);
        if ((int64_t)item >= total_items) break;
        int lo = 0, hi = n_jobs - 1;  // last job with item_begin <= item
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (jobs[mid].item_begin <= (int64_t)item) lo = mid;
            else hi = mid - 1;
        }
        const BatchJobDev &J = jobs[lo];
        shaft_item(J.b, J.rs, J.job, J.T_out, (int64_t)item - J.item_begin, status, sm[threadIdx.x >> 5]);
    }
}

int persistent_grid(const void *kernel) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 128, 0) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    return per_sm * rt_num_sms();
}

}  // namespace

extern "C" rt_status rt_trace_autotune(const rt_bvh *bvh, const rt_rayspec *rays, float *T_scratch,
                                       rt_trace_opts *opts, rt_stream_t stream) {
    if (!bvh || !rays || !opts || !T_scratch) return RT_ERR_INVALID_ARG;
    if (rays->kind == RT_RAYS_EXPLICIT || rays->ray_ids) return RT_ERR_UNSUPPORTED;
    RaySetDev rs;
    int64_t count = 0;
    RT_TRY(rt_rayset_dev(bvh, rays, &rs, &count));
    if (count == 0) return RT_OK;
    int dev = 0;
    cudaGetDevice(&dev);
    int log2n = 0;
    while ((1ll << (log2n + 1)) <= bvh->n) ++log2n;
    const TuneKey key{dev, log2n, rays->kind, rs.K, rays->kind == RT_RAYS_DIRS && rt_shaft_pays(bvh)};
    {
        std::lock_guard<std::mutex> g(g_tune_mu);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            opts->kernel = it->second.first;
            opts->order_block = it->second.second;
            return RT_OK;
        }
    }
    cudaStream_t st = (cudaStream_t)stream;
    unsigned long long *work = nullptr;
    RT_TRY(rt_alloc((void **)&work, 8 * kTuneBlocks, stream));
    const BvhDev b = bvh_dev(bvh);
    const int64_t ntiles = (bvh->n + 31) / 32;
    // about 4M rays per candidate: four contiguous blocks of tiles (all
    // directions of each tile) spread evenly over the Morton range, so the
    // sample sees several parts of the scene and each block keeps the
    // coherence of neighbouring tiles
    int64_t S = (1ll << 20) / (32ll * rs.K);
    if (S < 16) S = 16;
    int nb = kTuneBlocks;
    if (S * nb > ntiles) {
        nb = 1;
        S = ntiles;
    }
    const int blocks[] = {1, 16, 128, 1024};
    const int def_k = default_kernel(bvh, rays->kind);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f, def_ms = 1e30f;
    int best_k = def_k, best_b = 64, def_b = 64;
    rt_status res = RT_OK;
    for (int kernel = RT_KERNEL_RAY; kernel <= RT_KERNEL_RAY_REFILL && res == RT_OK; ++kernel) {
        const bool wide = kernel == RT_KERNEL_WIDE || kernel == RT_KERNEL_RAY_WIDE || kernel == RT_KERNEL_RAY_REFILL;
        // with a 4-wide tree the binary-tree strategies are not candidates (they
        // trail their 4-wide forms on every measured workload)
        if (wide != (bvh->n_wide > 0)) continue;
        // order_block only changes which rays share a warp for the packet strategies
        const int n_blocks = (kernel == RT_KERNEL_PACKET || kernel == RT_KERNEL_WIDE) ? 4 : 1;
        const int strat = kernel == RT_KERNEL_RAY_REFILL ? 5 : kernel == RT_KERNEL_RAY_WIDE ? 4 : kernel - 1;
        for (int bi = 0; bi < n_blocks && res == RT_OK; ++bi) {
            float ms = 1e30f;
            for (int rep = 0; rep < 2 && res == RT_OK; ++rep) {  // the first run warms caches
                cudaEventRecord(e0, st);
                for (int q = 0; q < nb && res == RT_OK; ++q) {
                    const bool shaft = kernel == RT_KERNEL_WIDE && rays->kind == RT_RAYS_DIRS;
                    TraceJob job = full_job(bvh, rs.K, blocks[bi], shaft);
                    // the same share of the scene in tiles of 32 and in shaft groups
                    const int64_t all = job.n_tiles, part = nb == 1 ? all : all * S / ntiles > 0 ? all * S / ntiles : 1;
                    job.n_tiles = part;
                    job.tile_base = nb == 1 ? 0 : (all - part) * (2 * q + 1) / (2 * nb);
                    if (job.order_block > part) job.order_block = (int32_t)part;
                    job.n_items = part * rs.K;
                    res = rt_trace_launch_job(b, rs, job, T_scratch, strat, stream, work + q);
                }
                cudaEventRecord(e1, st);
                float t = 0.f;
                if (cudaEventSynchronize(e1) != cudaSuccess) res = RT_ERR_CUDA;
                cudaEventElapsedTime(&t, e0, e1);
                if (rep > 0 && t < ms) ms = t;
            }
            if (res != RT_OK) break;
            if (ms < best) {
                best = ms;
                best_k = kernel;
                best_b = blocks[bi];
            }
            if (kernel == def_k && ms < def_ms) {
                def_ms = ms;
                def_b = blocks[bi];
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    rt_free(work, stream);
    if (res != RT_OK) return res;
    // another strategy replaces the default only when clearly faster: a
    // small margin on a sample is within run-to-run noise
    if (best_k != def_k && def_ms < 1e30f && best > kTuneMargin * def_ms) {
        best_k = def_k;
        best_b = def_b;
    }
    opts->kernel = best_k;
    opts->order_block = best_b;
    std::lock_guard<std::mutex> g(g_tune_mu);
    g_tune_cache[key] = {best_k, best_b};
    return RT_OK;
}

struct rt_batch {
    int n_jobs;
    int64_t n_rays, n_items;
    std::vector<int32_t> kernel, order_block;  // per job, in the caller's order
    void *table;                                // BatchJobDev[n_jobs] + work counter
    cudaGraph_t graph;
    cudaGraphExec_t exec;
};

extern "C" rt_status rt_batch_create(const rt_batch_job *jobs, int32_t n_jobs, int32_t autotune,
                                     rt_stream_t stream, rt_batch **out) {
    if (!out || !jobs || n_jobs <= 0 || n_jobs > 4096) return RT_ERR_INVALID_ARG;
    *out = nullptr;
    cudaStream_t st = (cudaStream_t)stream;
    std::vector<BatchJobDev> host(n_jobs);
    std::vector<double> cost(n_jobs);
    rt_batch *bt = new rt_batch();
    bt->n_jobs = n_jobs;
    bt->kernel.assign(n_jobs, 0);
    bt->order_block.assign(n_jobs, 0);
    bt->table = nullptr;
    bt->graph = nullptr;
    bt->exec = nullptr;
    for (int j = 0; j < n_jobs; ++j) {
        const rt_batch_job &J = jobs[j];
        int64_t count = 0;
        RaySetDev rs;
        rt_status r = (J.bvh && J.rays.kind != RT_RAYS_EXPLICIT && !J.rays.ray_ids)
                          ? rt_rayset_dev(J.bvh, &J.rays, &rs, &count)
                          : RT_ERR_INVALID_ARG;
        if (r == RT_OK && count > 0 && !J.T_out) r = RT_ERR_INVALID_ARG;
        if (r != RT_OK) {
            delete bt;
            return r;
        }
        rt_trace_opts o;
        memset(&o, 0, sizeof(o));
        o.kernel = default_kernel(J.bvh, J.rays.kind);
        o.order_block = 1;
        if (autotune && count > 0) {
            r = rt_trace_autotune(J.bvh, &J.rays, J.T_out, &o, stream);
            if (r != RT_OK) {
                delete bt;
                return r;
            }
        }
        bt->kernel[j] = o.kernel;
        bt->order_block[j] = o.order_block;
        BatchJobDev &H = host[j];
        memset(&H, 0, sizeof(H));
        H.b = bvh_dev(J.bvh);
        H.rs = rs;
        H.T_out = J.T_out;
        H.strat = o.kernel == RT_KERNEL_RAY_REFILL ? (J.bvh->n_wide > 0 ? 5 : 0)
                  : o.kernel == RT_KERNEL_RAY_WIDE ? (J.bvh->n_wide > 0 ? 4 : 0)
                  : o.kernel == RT_KERNEL_WIDE ? (J.bvh->n_wide > 0 ? (J.rays.kind == RT_RAYS_DIRS ? 3 : 2) : 1)
                  : o.kernel == RT_KERNEL_PACKET ? 1 : 0;
        H.job = full_job(J.bvh, rs.K, o.order_block, H.strat == 3);
        cost[j] = (double)count * log2((double)(J.bvh->n > 1 ? J.bvh->n : 2));
    }
    // a few shaft jobs of less than 2^17 rays together, beside other jobs: one
    // thread per ray in the others' kernel, since a launch of their own costs more
    // than they save (the four scenes of 2 to 7 thousand, tuned, the first of them
    // 48 thousand direction rays: 358 us with it in shafts, 315 without)
    int64_t shaft_rays = 0, other_rays = 0;
    for (int j = 0; j < n_jobs; ++j) (host[j].strat == 3 ? shaft_rays : other_rays) += host[j].job.n_out;
    if (other_rays > 0 && shaft_rays < (int64_t(1) << 17))
        for (int j = 0; j < n_jobs; ++j)
            if (host[j].strat == 3) {
                host[j].strat = 4;
                host[j].job = full_job(jobs[j].bvh, host[j].rs.K, 1, false);
                bt->kernel[j] = RT_KERNEL_RAY_WIDE;
                bt->order_block[j] = 1;
            }
    // shaft jobs (a queue and kernel of their own), item jobs, then lane-refill
    // jobs; largest estimated cost first in each
    std::vector<int> order(n_jobs);
    for (int j = 0; j < n_jobs; ++j) order[j] = j;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        auto rank = [&](int j) { return host[j].strat == 3 ? 0 : host[j].strat == 5 ? 2 : 1; };
        return rank(a) != rank(b) ? rank(a) < rank(b) : cost[a] > cost[b];
    });
    std::vector<BatchJobDev> queue(n_jobs);
    int64_t shafts = 0, items = 0, slots = 0, rays = 0;
    int n_shaft_jobs = 0, n_item_jobs = 0;
    for (int q = 0; q < n_jobs; ++q) {
        queue[q] = host[order[q]];
        if (queue[q].strat == 5) {
            queue[q].slot_begin = slots;
            slots += queue[q].job.n_items * 32;
        } else if (queue[q].strat == 3) {
            queue[q].item_begin = shafts;
            shafts += queue[q].job.n_items;
            ++n_shaft_jobs;
        } else {
            queue[q].item_begin = items;
            items += queue[q].job.n_items;
            ++n_item_jobs;
        }
        rays += queue[q].job.n_out;
    }
    bt->n_items = shafts + items + slots / 32;
    bt->n_rays = rays;
    const size_t tbytes = ((sizeof(BatchJobDev) * n_jobs + 255) & ~(size_t)255);
    rt_status r = rt_alloc(&bt->table, tbytes + 256, stream);
    if (r != RT_OK) {
        delete bt;
        return r;
    }
    BatchJobDev *dtab = (BatchJobDev *)bt->table;
    unsigned long long *work = (unsigned long long *)((char *)bt->table + tbytes);
    if (cudaMemcpyAsync(dtab, queue.data(), sizeof(BatchJobDev) * n_jobs, cudaMemcpyHostToDevice, st) !=
            cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        rt_free(bt->table, stream);
        delete bt;
        return RT_ERR_CUDA;
    }
    // capture: reset the queue counters, then one persistent launch for the item
    // and refill jobs and one for the shaft jobs, each on a branch of its own, so
    // that the second fills the multiprocessors as the blocks of the first leave.
    // The shaft jobs come second: their longest item is shorter than the others'
    // longest ray (four uniform scenes of 30 to 206 thousand Gaussians 61.1 ms, the
    // other way round 64.0)
    const int n_refill_jobs = n_jobs - n_shaft_jobs - n_item_jobs;
    cudaStream_t cap[2] = {nullptr, nullptr};
    cudaEvent_t ev[2] = {nullptr, nullptr};  // fork, join
    bool ok = true;
    for (int q = 0; q < 2; ++q)
        ok = ok && cudaStreamCreateWithFlags(&cap[q], cudaStreamNonBlocking) == cudaSuccess &&
             cudaEventCreateWithFlags(&ev[q], cudaEventDisableTiming) == cudaSuccess;
    int *status = rt_status_ptr();
    if (ok && (ok = cudaStreamBeginCapture(cap[0], cudaStreamCaptureModeThreadLocal) == cudaSuccess)) {
        cudaMemsetAsync(work, 0, 24, cap[0]);
        cudaEventRecord(ev[0], cap[0]);
        const BatchJobDev *rest = dtab + n_shaft_jobs;
        const int n_rest = n_item_jobs + n_refill_jobs;
        if (n_rest > 0) {
            cudaStreamWaitEvent(cap[1], ev[0], 0);
            if (n_refill_jobs == 0)
                k_trace_batch<false><<<persistent_grid((const void *)k_trace_batch<false>), 128, 0, cap[1]>>>(
                    rest, n_item_jobs, items, n_rest, slots, status, work);
            else if (n_item_jobs > 0)
                k_trace_batch<true><<<persistent_grid((const void *)k_trace_batch<true>), 128, 0, cap[1]>>>(
                    rest, n_item_jobs, items, n_rest, slots, status, work);
            else
                k_refill_batch<<<persistent_grid((const void *)k_refill_batch), 128, 0, cap[1]>>>(
                    rest, n_refill_jobs, slots, status, work + 1);
            cudaEventRecord(ev[1], cap[1]);
        }
        if (n_shaft_jobs > 0)
            k_shaft_batch<<<persistent_grid((const void *)k_shaft_batch), 128, 0, cap[0]>>>(dtab, n_shaft_jobs, shafts,
                                                                                            status, work + 2);
        if (n_rest > 0) cudaStreamWaitEvent(cap[0], ev[1], 0);
        ok = cudaStreamEndCapture(cap[0], &bt->graph) == cudaSuccess;
    }
    if (ok) ok = cudaGraphInstantiate(&bt->exec, bt->graph, 0) == cudaSuccess;
    for (int q = 0; q < 2; ++q) {
        if (ev[q]) cudaEventDestroy(ev[q]);
        if (cap[q]) cudaStreamDestroy(cap[q]);
    }
    if (!ok) {
        cudaGetLastError();
        if (bt->exec) cudaGraphExecDestroy(bt->exec);
        if (bt->graph) cudaGraphDestroy(bt->graph);
        rt_free(bt->table, stream);
        delete bt;
        return RT_ERR_CUDA;
    }
    *out = bt;
    return RT_OK;
}

extern "C" rt_status rt_batch_run(rt_batch *bt, rt_stream_t stream) {
    if (!bt) return RT_ERR_INVALID_ARG;
    return cudaGraphLaunch(bt->exec, (cudaStream_t)stream) == cudaSuccess ? RT_OK : RT_ERR_CUDA;
}

extern "C" rt_status rt_batch_info(const rt_batch *bt, int64_t *n_rays, int64_t *n_items, int32_t *kernel,
                                   int32_t *order_block) {
    if (!bt) return RT_ERR_INVALID_ARG;
    if (n_rays) *n_rays = bt->n_rays;
    if (n_items) *n_items = bt->n_items;
    for (int j = 0; j < bt->n_jobs; ++j) {
        if (kernel) kernel[j] = bt->kernel[j];
        if (order_block) order_block[j] = bt->order_block[j];
    }
    return RT_OK;
}

extern "C" rt_status rt_batch_destroy(rt_batch *bt, rt_stream_t stream) {
    if (!bt) return RT_ERR_INVALID_ARG;
    cudaStreamSynchronize((cudaStream_t)stream);
    if (bt->exec) cudaGraphExecDestroy(bt->exec);
    if (bt->graph) cudaGraphDestroy(bt->graph);
    rt_free(bt->table, stream);
    delete bt;
    return RT_OK;
}
