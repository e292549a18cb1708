// rt_build.cu -- LBVH construction on the device (Sec. 4.1: a binary radix
// tree over the Gaussians in the manner of Karras 2012, leaves = tight boxes
// of single Gaussians, internal nodes = union of their children).
//
// Steps (all kernels below, one stream, one synchronisation at the end):
//   k_bounds       input check and per-axis min/max of the means
//   k_morton       30-bit Morton codes, float32 IEEE quantisation (no FMA)
//   k_sort_small   both for up to 12288 Gaussians, by counting
//   k_radix_*      stable LSD radix sort of (code, index), 8-bit digits, 4 passes
//   k_prep         permutation, inverse permutation, 64-bit keys code<<32|index,
//                  per-Gaussian record (mean, opacity, whitening W = S^-1 R^T)
//                  and its leaf box, in sorted order
//   k_topology     internal-node children by the longest-common-prefix split;
//                  in other blocks of the launch the shaft groups
//   k_refit        bottom-up child boxes: within a block of leaves in shared
//                  memory, across blocks the second thread to reach a node
//                  (atomic arrival count) forms its box and climbs on
//   k_wide         the 4-wide tree: every binary node as if it were the root of
//                  a wide node, all at once
// What a build costs is launches and dependent loads, not bytes.
#include <math.h>
#include <string.h>

#include "rt_internal.cuh"

namespace {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;

__device__ __forceinline__ uint32_t f2ord(float f) {
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Records a failed input check in the status word (asynchronous callers).
__global__ void k_report_invalid(const unsigned *bad, int *status) {
    if (*bad) rt_set_error(status, RT_ERR_INVALID_ARG);
}

// Scene words (zero before the build): [0..2] the complement of the ordered
// minimum of the means, [3..5] the ordered maximum, [6] non-zero if the input
// check failed, [7] shaft groups, [8] levels of the binary tree.
enum { SCN_BAD = 6, SCN_GROUPS = 7, SCN_LEVELS = 8, SCN_WORDS = 9, SCN_BYTES = 256 };
__device__ __forceinline__ float scene_lo(const uint32_t *scn, int c) { return ord2f(~scn[c]); }
__device__ __forceinline__ float scene_hi(const uint32_t *scn, int c) { return ord2f(scn[3 + c]); }

// Input check (every value finite, scales > 0, a non-zero quaternion, opacity
// in [0, 1]) and bounds of the means.  The blocks' results meet in six words:
// two blocks per multiprocessor, since one atomic per warp of a full grid on
// the same word took 40 us at 300k Gaussians.
__global__ void __launch_bounds__(512) k_bounds(const float *__restrict__ mean, const float *__restrict__ scale,
                                                const float *__restrict__ quat, const float *__restrict__ opacity,
                                                int64_t n, uint32_t *scn) {
    __shared__ uint32_t red[6];
    if (threadIdx.x < 6) red[threadIdx.x] = 0u;
    __syncthreads();
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    bool ok = true;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        float qn = 0.0f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float m = mean[3 * i + c], sc = scale[3 * i + c];
            ok = ok && isfinite(m) && isfinite(sc) && sc > 0.0f;
            lo[c] = fminf(lo[c], m);
            hi[c] = fmaxf(hi[c], m);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float q = quat[4 * i + c];
            ok = ok && isfinite(q);
            qn += q * q;
        }
        const float o = opacity[i];
        ok = ok && qn > 0.0f && o >= 0.0f && o <= 1.0f;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const uint32_t l = __reduce_max_sync(0xffffffffu, ~f2ord(lo[c])), h = __reduce_max_sync(0xffffffffu, f2ord(hi[c]));
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&red[c], l);
            atomicMax(&red[3 + c], h);
        }
    }
    if (!ok) atomicOr(scn + SCN_BAD, 1u);
    __syncthreads();
    if (threadIdx.x < 6) atomicMax(scn + threadIdx.x, red[threadIdx.x]);
}

__device__ __forceinline__ uint32_t spread10(uint32_t v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// Quantisation with separately rounded float32 operations:
// u = (mu - lo) / (hi - lo), q = clamp(floor(u * 1024), 0, 1023); 0 if hi == lo.
__device__ __forceinline__ uint32_t morton_code(const float *__restrict__ m, const float (&lo)[3], const float (&ext)[3]) {
    uint32_t q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (ext[c] == 0.0f) {
            q[c] = 0;
            continue;
        }
        float u = __fdiv_rn(__fsub_rn(m[c], lo[c]), ext[c]);
        float v = __fmul_rn(u, 1024.0f);
        int qi = (int)floorf(v);
        qi = qi < 0 ? 0 : (qi > 1023 ? 1023 : qi);
        q[c] = (uint32_t)qi;
    }
    return (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
}
// The scene's bounds from the scene words; one thread writes them out.
__device__ __forceinline__ void scene_bounds(const uint32_t *scn, float *bounds_out, float (&lo)[3], float (&ext)[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        lo[c] = scene_lo(scn, c);
        float hi = scene_hi(scn, c);
        ext[c] = __fsub_rn(hi, lo[c]);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            bounds_out[c] = lo[c];
            bounds_out[3 + c] = hi;
        }
    }
}
__global__ void k_morton(const float *__restrict__ mean, int64_t n, const uint32_t *scn,
                         float *bounds_out, uint32_t *codes, int32_t *vals) {
    float lo[3], ext[3];
    scene_bounds(scn, bounds_out, lo, ext);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        codes[i] = morton_code(mean + 3 * i, lo, ext);
        vals[i] = (int32_t)i;
    }
}

// counts[d * nblk + b] = number of keys of tile b (kSortThreads * ITEMS keys)
// with digit d
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint32_t *__restrict__ keys,
                                                             int64_t n, int shift, int nblk,
                                                             uint32_t *counts) {
    __shared__ uint32_t hist[kRadix];
    const int64_t base = (int64_t)blockIdx.x * (kSortThreads * ITEMS) + threadIdx.x;
    uint32_t k[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) k[it] = base + it * kSortThreads < n ? keys[base + it * kSortThreads] : 0u;
    for (int d = threadIdx.x; d < kRadix; d += kSortThreads) hist[d] = 0;
    __syncthreads();
#pragma unroll
    for (int it = 0; it < ITEMS; ++it)
        if (base + it * kSortThreads < n) atomicAdd(&hist[(k[it] >> shift) & (kRadix - 1)], 1u);
    __syncthreads();
    for (int d = threadIdx.x; d < kRadix; d += kSortThreads) counts[(int64_t)d * nblk + blockIdx.x] = hist[d];
}

// Per digit (one block each) the exclusive scan over the tiles of its counts,
// in place, and their total.  The scan over the digits is left to the scatter.
// (One block scanning all counts took 31 us a pass at 300k keys; segment sums,
// their scan and a scan per segment 14 us in three launches.)
__global__ void __launch_bounds__(256) k_radix_scan(uint32_t *counts, int nblk, uint32_t *totals) {
    __shared__ uint32_t ws[8];
    uint32_t *row = counts + (int64_t)blockIdx.x * nblk;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    uint32_t carry = 0;
    for (int b0 = 0; b0 < nblk; b0 += 1024) {
        uint32_t v[4], sum = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = b0 + 4 * t + k;
            v[k] = i < nblk ? row[i] : 0u;
            sum += v[k];
        }
        uint32_t inc = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += u;
        }
        if (lane == 31) ws[w] = inc;
        __syncthreads();
        uint32_t run = carry + inc - sum, all = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k < w) run += ws[k];
            all += ws[k];
        }
        carry += all;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = b0 + 4 * t + k;
            if (i < nblk) row[i] = run;
            run += v[k];
        }
        __syncthreads();
    }
    if (t == 0) totals[blockIdx.x] = carry;
}

// Stable ranks of a warp's ITEMS * 32 consecutive keys among its own keys of
// equal digit, in index order (round, lane); cnt[d] (zero before) ends as the
// warp's count of digit d.  Keys with live[] false take no part.
template <int ITEMS>
__device__ __forceinline__ void warp_ranks(const uint32_t (&key)[ITEMS], const bool (&live)[ITEMS], int shift,
                                           uint32_t *cnt, uint32_t (&rank)[ITEMS]) {
    const uint32_t lt_mask = (1u << (threadIdx.x & 31)) - 1u;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const uint32_t d = live[it] ? ((key[it] >> shift) & (kRadix - 1)) : 0xffffffffu;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t r = __popc(peers & lt_mask), c = live[it] ? cnt[d] : 0u;
        __syncwarp();
        if (live[it] && r == 0) cnt[d] = c + __popc(peers);
        __syncwarp();
        rank[it] = c + r;
    }
}

// Stable scatter of a tile: each warp ranks its own consecutive keys, then the
// warps' counts are summed once (two block barriers a tile; ranking round by
// round over the whole block took four a round, 21 us a pass at any size up
// to 300k).
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_radix_scatter(
    const uint32_t *__restrict__ keys_in, const int32_t *__restrict__ vals_in, int64_t n, int shift,
    int nblk, const uint32_t *__restrict__ offsets, const uint32_t *__restrict__ totals, uint32_t *keys_out,
    int32_t *vals_out) {
    __shared__ uint32_t wcnt[kSortWarps][kRadix];
    __shared__ uint32_t ws[kSortWarps];
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const int64_t base = (int64_t)blockIdx.x * (kSortThreads * ITEMS) + w * (32 * ITEMS) + lane;
    uint32_t key[ITEMS], rank[ITEMS];
    int32_t val[ITEMS];
    bool live[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        live[it] = base + 32 * it < n;
        key[it] = live[it] ? keys_in[base + 32 * it] : 0u;
        val[it] = live[it] ? vals_in[base + 32 * it] : 0;
    }
    for (int j = t; j < kSortWarps * kRadix; j += kSortThreads) (&wcnt[0][0])[j] = 0;
    // one digit a thread: keys of smaller digits, then of this one in tiles before
    const uint32_t tot = totals[t];
    uint32_t run = offsets[(int64_t)t * nblk + blockIdx.x], inc = tot;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += u;
    }
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    run += inc - tot;
#pragma unroll
    for (int k = 0; k < kSortWarps; ++k)
        if (k < w) run += ws[k];
    warp_ranks<ITEMS>(key, live, shift, wcnt[w], rank);
    __syncthreads();
#pragma unroll
    for (int ww = 0; ww < kSortWarps; ++ww) {
        const uint32_t c = wcnt[ww][t];
        wcnt[ww][t] = run;
        run += c;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        if (!live[it]) continue;
        const uint32_t pos = wcnt[w][(key[it] >> shift) & (kRadix - 1)] + rank[it];
        keys_out[pos] = key[it];
        vals_out[pos] = val[it];
    }
}
static_assert(kSortThreads == kRadix, "one digit a thread");

// Morton codes of a small scene in sorted order (ties by index) without a sort:
// every block forms all codes in shared memory, and the place of one is how
// many are smaller, or equal with a smaller index; a warp counts for each.
// n^2 compares, but no chain: four radix passes in one block took 26 us at
// 4096 Gaussians, and k_morton before them 4 us more; this 10 us (18 with 8
// threads a code, which form 16 codes each one after the other).
// Builds of 8192 Gaussians take 112 us so and 154 with the radix sort, of 12288
// (48 KB of codes) 149 and 157.
constexpr int kSmallSort = 12288;
__global__ void __launch_bounds__(1024) k_sort_small(const float *__restrict__ mean, int n, const uint32_t *scn,
                                                     float *bounds_out, uint32_t *codes, int32_t *vals) {
    __shared__ uint4 sk4[kSmallSort / 4];
    uint32_t *sk = reinterpret_cast<uint32_t *>(sk4);
    float lo[3], ext[3];
    scene_bounds(scn, bounds_out, lo, ext);
    const int padded = (n + 127) / 128 * 128;
#pragma unroll 4
    for (int i = threadIdx.x; i < padded; i += 1024) sk[i] = i < n ? morton_code(mean + 3 * i, lo, ext) : 0xffffffffu;
    __syncthreads();
    const int e = blockIdx.x * 32 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t key = sk[e];
    int cnt = 0;
#pragma unroll 4
    for (int j = lane; j < padded / 4; j += 32) {
        const uint4 v = sk4[j];
        const int d = e - 4 * j;  // the first d of the four have a smaller index
        cnt += (v.x < key + (d > 0)) + (v.y < key + (d > 1)) + (v.z < key + (d > 2)) + (v.w < key + (d > 3));
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0 && e < n) {
        codes[cnt] = key;
        vals[cnt] = e;
    }
}

// Per-Gaussian record and leaf box in sorted order; with the sorted codes (a
// build) also the permutation (perm = the sort's values), its inverse and the
// keys.
__global__ void k_prep(const float *__restrict__ mean, const float *__restrict__ scale,
                       const float *__restrict__ quat, const float *__restrict__ opacity,
                       const int32_t *__restrict__ perm, const uint32_t *__restrict__ codes, int64_t n, rt_params prm,
                       const uint32_t *scn, float4 *gauss, float *leafbox, int32_t *perm_out, int32_t *rank,
                       uint64_t *keys) {
    // absolute box margin: 1e-6 of the scene's coordinate scale
    float L = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float lo = scene_lo(scn, c), hi = scene_hi(scn, c);
        L = fmaxf(L, fmaxf(fabsf(lo), fmaxf(fabsf(hi), hi - lo)));
    }
    const float margin = 1e-6f * L;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        int32_t i = perm[p];
        if (codes) {
            perm_out[p] = i;
            rank[i] = (int32_t)p;
            keys[p] = ((uint64_t)codes[p] << 32) | (uint32_t)i;
        }
        float qw = quat[4 * i], qx = quat[4 * i + 1], qy = quat[4 * i + 2], qz = quat[4 * i + 3];
        float qn = sqrtf(qw * qw + qx * qx + qy * qy + qz * qz);
        qw /= qn; qx /= qn; qy /= qn; qz /= qn;
        float R[3][3];
        R[0][0] = 1.f - 2.f * (qy * qy + qz * qz); R[0][1] = 2.f * (qx * qy - qw * qz); R[0][2] = 2.f * (qx * qz + qw * qy);
        R[1][0] = 2.f * (qx * qy + qw * qz); R[1][1] = 1.f - 2.f * (qx * qx + qz * qz); R[1][2] = 2.f * (qy * qz - qw * qx);
        R[2][0] = 2.f * (qx * qz - qw * qy); R[2][1] = 2.f * (qy * qz + qw * qx); R[2][2] = 1.f - 2.f * (qx * qx + qy * qy);
        float s[3] = {scale[3 * i], scale[3 * i + 1], scale[3 * i + 2]};
        float mu[3] = {mean[3 * i], mean[3 * i + 1], mean[3 * i + 2]};
        float o = opacity[i];
        float W[3][3];  // row k = column k of R divided by s_k
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) W[k][c] = __fdiv_rn(R[c][k], s[k]);
        gauss[4 * p + 0] = make_float4(mu[0], mu[1], mu[2], o);
        gauss[4 * p + 1] = make_float4(W[0][0], W[0][1], W[0][2], __int_as_float(i));
        gauss[4 * p + 2] = make_float4(W[1][0], W[1][1], W[1][2], 0.f);
        gauss[4 * p + 3] = make_float4(W[2][0], W[2][1], W[2][2], 0.f);
        // support radius: k_sigma, or the opacity-aware radius (same accepted set)
        float K = prm.k_sigma;
        bool empty = false;
        if (prm.box_mode == 1) {
            if (o < prm.alpha_min) empty = true;
            else {
                float kk = 2.0f * logf(o / prm.alpha_min);
                kk = kk * (1.0f + 1e-4f) + 1e-6f;  // outward margin for logf rounding
                if (kk < K * K) K = sqrtf(kk);
            }
        }
        float *bx = leafbox + 6 * p;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            // half-extent along world axis c: K sqrt(sum_k (R_ck s_k)^2), widened by
            // 1e-4 relative plus a few ulps of |mu| so the float box contains the
            // exact support and the slab test never misses an accepted peak
            float a0 = R[c][0] * s[0], a1 = R[c][1] * s[1], a2 = R[c][2] * s[2];
            float h = K * sqrtf(a0 * a0 + a1 * a1 + a2 * a2);
            h = h * (1.0f + 1e-4f) + 4.0f * 1.1920929e-7f * fabsf(mu[c]) + margin + 1e-30f;
            bx[c] = empty ? __int_as_float(0x7fc00000) : __fsub_rd(mu[c], h);
            bx[3 + c] = empty ? __int_as_float(0x7fc00000) : __fadd_ru(mu[c], h);
        }
    }
}

// Shaft groups: each tile of 64 sorted positions is cut where its means lie
// far apart (a jump of the Morton curve), since a packet of a direction set
// walks the tree once per group with the box of the group's means.  A walk's
// cost is taken as SA(box + one leaf) (10 + 0.27 rays): the Gaussians a shaft
// of that box meets, times the issue slots one of them costs the walk and one
// ray.  The cut of the largest gain is made first, until none gains.  One
// warp per tile, lane l holds positions 2 l and 2 l + 1; the boxes left and
// right of every cut come from two segmented scans.  The order of the list is
// that of the tiles' arrival.
struct Box6 {
    float l[3], h[3];
};
__device__ __forceinline__ Box6 box_join(const Box6 &a, const Box6 &b) {
    Box6 r;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        r.l[c] = fminf(a.l[c], b.l[c]);
        r.h[c] = fmaxf(a.h[c], b.h[c]);
    }
    return r;
}
template <bool UP>
__device__ __forceinline__ Box6 box_shfl(const Box6 &a, int off) {
    Box6 r;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        r.l[c] = UP ? __shfl_up_sync(0xffffffffu, a.l[c], off) : __shfl_down_sync(0xffffffffu, a.l[c], off);
        r.h[c] = UP ? __shfl_up_sync(0xffffffffu, a.h[c], off) : __shfl_down_sync(0xffffffffu, a.h[c], off);
    }
    return r;
}
__device__ __forceinline__ void tile_groups(const float4 *__restrict__ gauss, const float *__restrict__ leafbox,
                                            int64_t n, int2 *groups, unsigned *n_groups, int64_t warp0, int64_t warps) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t tiles = (n + 63) / 64;
    for (int64_t tile = warp0; tile < tiles; tile += warps) {
        const int64_t left = n - tile * 64;
        const int cnt = (int)(left < 64 ? left : 64);
        Box6 v[2];
        float L[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const bool in = 2 * lane + r < cnt;
            const int64_t p = tile * 64 + (in ? 2 * lane + r : 0);
            const float4 g = gauss[4 * p];
            const float m[3] = {g.x, g.y, g.z};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[r].l[c] = in ? m[c] : INFINITY;
                v[r].h[c] = in ? m[c] : -INFINITY;
                const float e = leafbox[6 * p + 3 + c] - leafbox[6 * p + c];
                if (in && e == e) L[c] += e / (float)cnt;  // an empty box is NaN
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
            for (int off = 16; off > 0; off >>= 1) L[c] += __shfl_xor_sync(FULL, L[c], off);
        const Box6 both = box_join(v[0], v[1]);
        uint64_t starts = 1ull | (cnt < 64 ? 1ull << cnt : 0ull);  // the end of a short tile closes its last group
        for (int it = 0; it < 63; ++it) {
            const bool sa = (starts >> (2 * lane)) & 1ull, sb = (starts >> (2 * lane + 1)) & 1ull;
            const bool sn = lane == 31 || ((starts >> (2 * lane + 2)) & 1ull);
            // pre: the box from the group's start through position 2 l + 1;
            // suf: from position 2 l to the group's end
            Box6 pre = sb ? v[1] : both, suf = sb ? v[0] : both;
            int fp = sa || sb, fs = sb || sn;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const Box6 a = box_shfl<true>(pre, off), z = box_shfl<false>(suf, off);
                const int ap = __shfl_up_sync(FULL, fp, off), zs = __shfl_down_sync(FULL, fs, off);
                if (lane >= off && !fp) {
                    pre = box_join(pre, a);
                    fp = ap;
                }
                if (lane + off < 32 && !fs) {
                    suf = box_join(suf, z);
                    fs = zs;
                }
            }
            const Box6 prv = box_shfl<true>(pre, 1), nxt = box_shfl<false>(suf, 1);
            auto cost = [&](const Box6 &x, int rays) {
                const float dx = x.h[0] - x.l[0] + L[0], dy = x.h[1] - x.l[1] + L[1], dz = x.h[2] - x.l[2] + L[2];
                return (dx * dy + dy * dz + dz * dx) * (10.0f + 0.27f * (float)rays);
            };
            float gain = 0.0f;
            int at = 0;
#pragma unroll
            for (int r = 0; r < 2; ++r) {  // the cut in front of position 2 l + r
                const int c = 2 * lane + r;
                if (c == 0 || c >= cnt || (r ? sb : sa)) continue;
                const uint64_t below = starts & ((1ull << c) - 1ull), above = starts >> c;
                const int s0 = 63 - __clzll((long long)below), s1 = above ? c + __ffsll((long long)above) - 1 : cnt;
                const Box6 A = r == 0 ? prv : sa ? v[0] : box_join(prv, v[0]);
                const Box6 B = r == 0 ? suf : sn ? v[1] : box_join(nxt, v[1]);
                const float g = cost(box_join(A, B), s1 - s0) - cost(A, c - s0) - cost(B, s1 - c);
                if (g > gain) {
                    gain = g;
                    at = c;
                }
            }
            const uint32_t key = __float_as_uint(gain), best = __reduce_max_sync(FULL, key);
            if (best == 0u) break;
            starts |= 1ull << __shfl_sync(FULL, at, __ffs(__ballot_sync(FULL, key == best)) - 1);
        }
        unsigned slot = 0;
        const uint64_t own = cnt < 64 ? starts & ((1ull << cnt) - 1ull) : starts;
        if (lane == 0) slot = atomicAdd(n_groups, (unsigned)__popcll(own));
        slot = __shfl_sync(FULL, slot, 0);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int c = 2 * lane + r;
            if (!((own >> c) & 1ull)) continue;
            const uint64_t above = c < 63 ? starts >> (c + 1) : 0ull;
            const int s1 = above ? c + __ffsll((long long)above) : cnt;
            groups[slot + __popcll(own & ((1ull << c) - 1ull))] = make_int2((int)(tile * 64 + c), s1 - c);
        }
    }
}

__device__ __forceinline__ int lcp(const uint64_t *keys, int64_t n, int64_t i, int64_t j) {
    if (j < 0 || j >= n) return -1;
    return __clzll(keys[i] ^ keys[j]);
}

// Internal node i: direction d toward the longer common prefix, range end j
// by exponential + binary search, split gamma by binary search; children
// gamma and gamma+1 are leaves when they are the range's ends.
// Also the node's range of sorted positions, and zero for its arrival count.
__device__ __forceinline__ void karras(const uint64_t *__restrict__ keys, int64_t n, float4 *nodes, int32_t *parent,
                                       uint32_t *arrivals, int64_t i0, int64_t step) {
    for (int64_t i = i0; i < n - 1; i += step) {
        int d = (lcp(keys, n, i, i + 1) - lcp(keys, n, i, i - 1)) >= 0 ? 1 : -1;
        int dmin = lcp(keys, n, i, i - d);
        int64_t lmax = 2;
        while (lcp(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;
        int64_t l = 0;
        for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
            if (lcp(keys, n, i, i + (l + t) * d) > dmin) l += t;
        int64_t j = i + l * d;
        int dnode = lcp(keys, n, i, j);
        int64_t s = 0, t = l;
        for (;;) {
            t = (t + 1) >> 1;
            if (lcp(keys, n, i, i + (s + t) * d) > dnode) s += t;
            if (t == 1) break;
        }
        int64_t gamma = i + s * d + (d < 0 ? -1 : 0);
        int64_t first = i < j ? i : j, last = i < j ? j : i;
        uint32_t lref, rref;
        if (first == gamma) {
            lref = RT_LEAF_BIT | (uint32_t)gamma;
            parent[(n - 1) + gamma] = (int32_t)i;
        } else {
            lref = (uint32_t)gamma;
            parent[gamma] = (int32_t)i;
        }
        if (last == gamma + 1) {
            rref = RT_LEAF_BIT | (uint32_t)(gamma + 1);
            parent[(n - 1) + gamma + 1] = (int32_t)i;
        } else {
            rref = (uint32_t)(gamma + 1);
            parent[gamma + 1] = (int32_t)i;
        }
        nodes[4 * i + 3] = make_float4(__uint_as_float(lref), __uint_as_float(rref), __int_as_float((int)first),
                                       __int_as_float((int)last));
        arrivals[i] = 0u;
        if (i == 0) parent[0] = -1;
    }
}

// The tree's topology in the first kblocks blocks, the shaft groups (which
// need the same inputs and are a chain of warp scans of their own, 12 us at
// any small size) in the others.
__global__ void __launch_bounds__(128) k_topology(const uint64_t *__restrict__ keys, int64_t n, float4 *nodes,
                                                  int32_t *parent, uint32_t *arrivals, int kblocks,
                                                  const float4 *__restrict__ gauss, const float *__restrict__ leafbox,
                                                  int2 *groups, unsigned *n_groups) {
    if ((int)blockIdx.x < kblocks)
        karras(keys, n, nodes, parent, arrivals, blockIdx.x * 128ll + threadIdx.x, kblocks * 128ll);
    else
        tile_groups(gauss, leafbox, n, groups, n_groups, (blockIdx.x - kblocks) * 4ll + (threadIdx.x >> 5),
                    ((int)gridDim.x - kblocks) * 4ll);
}

__device__ __forceinline__ void store_child_box(float4 *nodes, int32_t node, bool right, const float b[6]) {
    float2 *nd = reinterpret_cast<float2 *>(nodes + 4 * (int64_t)node) + (right ? 3 : 0);
    __stcg(nd, make_float2(b[0], b[3]));
    __stcg(nd + 1, make_float2(b[1], b[4]));
    __stcg(nd + 2, make_float2(b[2], b[5]));
}

// One thread per leaf climbs toward the root.  At each internal node it
// stores its subtree's box into the node's child slot and bumps the node's
// arrival count: the first arrival stops, the second (which then sees both
// slots) forms the union and continues.  No thread ever waits for another's
// arrival.  A node whose range lies within the block's leaves (all but one in
// kRefitLeaves) keeps its boxes and count in shared memory, where a level
// costs a fraction of the atomic through L2 and what orders it.  The counts
// carry the first arrival's height (count in the low 8 bits), so the root's
// height comes out for free: the levels of the tree.
// Up to 4096 leaves (CLUSTER) all blocks form one cluster, and the nodes that
// straddle blocks are in the shared memory of the block their index lies in:
// 4096 leaves 23.4 us through L2, 15.3 so.
__device__ __forceinline__ uint32_t atomic_add_acq_rel(uint32_t *p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
// Thread-block clusters: a barrier of all blocks, the address of `p` in block
// `rank`'s shared memory, and a counter there.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
template <class T>
__device__ __forceinline__ T *cluster_map(T *p, int rank) {
    uint64_t a;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(a) : "l"((uint64_t)p), "r"(rank));
    return reinterpret_cast<T *>(a);
}
__device__ __forceinline__ uint32_t atomic_add_acq_rel_cluster(uint32_t *p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.acq_rel.cluster.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
constexpr int kRefitLeaves = 512;
template <bool CLUSTER>
__global__ void __launch_bounds__(kRefitLeaves) k_refit(const float *__restrict__ leafbox,
                                                        const int32_t *__restrict__ parent, int64_t n, float4 *nodes,
                                                        uint32_t *arrivals, uint32_t *levels) {
    __shared__ float box[kRefitLeaves][12];
    __shared__ float4 ref[kRefitLeaves];
    __shared__ int32_t par[kRefitLeaves];
    __shared__ uint32_t cnt[kRefitLeaves];
    const int t = threadIdx.x;
    // the grid has no block beyond the leaves, a cluster may: those go round once
    // too, for its barriers
    int64_t b0 = (int64_t)blockIdx.x * kRefitLeaves;
    do {
        const int64_t p = b0 + t, b1 = b0 + kRefitLeaves < n ? b0 + kRefitLeaves : n;
        const float4 none = make_float4(0.f, 0.f, __int_as_float(-1), __int_as_float(0x7fffffff));
        ref[t] = p < n - 1 ? __ldcg(nodes + 4 * p + 3) : none;
        par[t] = p < n - 1 ? parent[p] : -1;
        cnt[t] = 0u;
        float b[6];
        int32_t node = -1;
        if (p < n) {
#pragma unroll
            for (int c = 0; c < 6; ++c) b[c] = leafbox[6 * p + c];
            node = parent[(n - 1) + p];
        }
        uint32_t child = RT_LEAF_BIT | (uint32_t)p, height = 0u;
        if constexpr (CLUSTER) cluster_sync();  // every block's slots are ready
        auto local = [&](const float4 &r) { return __float_as_int(r.z) >= b0 && __float_as_int(r.w) < b1; };
        __syncthreads();
        while (node >= 0 && node >= b0 && node < b1) {
            const int q = (int)(node - b0);
            const float4 r = ref[q];
            if (!local(r)) break;
            float *nd = box[q] + (__float_as_uint(r.x) != child ? 6 : 0);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                nd[2 * c] = b[c];
                nd[2 * c + 1] = b[3 + c];
            }
            __threadfence_block();
            const uint32_t old = atomicAdd(&cnt[q], 1u + (height << 8));
            if (old == 0u) {
                node = -1;
                break;
            }
            height = max(height, old >> 8) + 1u;
            __threadfence_block();
            const volatile float *l = box[q];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                b[c] = fminf(l[2 * c], l[6 + 2 * c]);
                b[3 + c] = fmaxf(l[2 * c + 1], l[7 + 2 * c]);
            }
            child = (uint32_t)node;
            if (node == 0) *levels = height;
            node = par[q];
        }
        if constexpr (CLUSTER) {
            while (node >= 0) {
                const int own = (int)(node / kRefitLeaves), q = (int)(node % kRefitLeaves);
                const float4 r = *cluster_map(&ref[q], own);
                const int up = *cluster_map(&par[q], own);
                float *x = cluster_map(&box[q][0], own), *nd = x + (__float_as_uint(r.x) != child ? 6 : 0);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    nd[2 * c] = b[c];
                    nd[2 * c + 1] = b[3 + c];
                }
                const uint32_t old = atomic_add_acq_rel_cluster(cluster_map(&cnt[q], own), 1u + (height << 8));
                if (old == 0u) break;
                height = max(height, old >> 8) + 1u;
                const volatile float *l = x;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    b[c] = fminf(l[2 * c], l[6 + 2 * c]);
                    b[3 + c] = fmaxf(l[2 * c + 1], l[7 + 2 * c]);
                }
                child = (uint32_t)node;
                if (node == 0) *levels = height;
                node = up;
            }
            cluster_sync();  // no block leaves while another may reach into it
        } else {
            while (node >= 0) {
                const float4 r = __ldcg(nodes + 4 * (int64_t)node + 3);
                store_child_box(nodes, node, __float_as_uint(r.x) != child, b);
                const uint32_t old = atomic_add_acq_rel(&arrivals[node], 1u + (height << 8));
                if (old == 0u) break;
                height = max(height, old >> 8) + 1u;
                const float4 *nd = nodes + 4 * (int64_t)node;
                const float4 x = __ldcg(nd), y = __ldcg(nd + 1), z = __ldcg(nd + 2);
                // slots: (L.lo.x, L.hi.x, L.lo.y, L.hi.y, L.lo.z, L.hi.z, R.lo.x, ...)
                b[0] = fminf(x.x, y.z); b[3] = fmaxf(x.y, y.w);
                b[1] = fminf(x.z, z.x); b[4] = fmaxf(x.w, z.y);
                b[2] = fminf(y.x, z.z); b[5] = fmaxf(y.y, z.w);
                child = (uint32_t)node;
                if (node == 0) *levels = height;
                node = parent[node];
            }
        }
        __syncthreads();
        if (p < n - 1 && (CLUSTER || local(ref[t]))) {
            const float *l = box[t];
            float4 *nd = nodes + 4 * p;
            nd[0] = make_float4(l[0], l[1], l[2], l[3]);
            nd[1] = make_float4(l[4], l[5], l[6], l[7]);
            nd[2] = make_float4(l[8], l[9], l[10], l[11]);
        }
        __syncthreads();
        b0 += (int64_t)gridDim.x * kRefitLeaves;
    } while (!CLUSTER && b0 < n);
}

// Surface area of a box stored (lo.x, hi.x, lo.y, hi.y, lo.z, hi.z); -1 for NaN.
__device__ __forceinline__ float box_area(const float b[6]) {
    const float dx = b[1] - b[0], dy = b[3] - b[2], dz = b[5] - b[4];
    const float a = dx * dy + dy * dz + dz * dx;
    return a == a ? a : -1.0f;
}

// One child slot of a wide node under construction.
struct WideSlot {
    uint32_t ref;
    float b[6];  // (lo.x, hi.x, lo.y, hi.y, lo.z, hi.z)
    float area;  // surface area of an internal child (-1: NaN box), -2: leaf or none
};
__device__ __forceinline__ void wide_children(const float4 *__restrict__ nodes, int32_t e, WideSlot &l, WideSlot &r) {
    const float4 a = nodes[4 * (int64_t)e], c = nodes[4 * (int64_t)e + 1], d = nodes[4 * (int64_t)e + 2],
                 f = nodes[4 * (int64_t)e + 3];
    l.ref = __float_as_uint(f.x);
    l.b[0] = a.x; l.b[1] = a.y; l.b[2] = a.z; l.b[3] = a.w; l.b[4] = c.x; l.b[5] = c.y;
    r.ref = __float_as_uint(f.y);
    r.b[0] = c.z; r.b[1] = c.w; r.b[2] = d.x; r.b[3] = d.y; r.b[4] = d.z; r.b[5] = d.w;
    l.area = (l.ref & RT_LEAF_BIT) ? -2.0f : box_area(l.b);
    r.area = (r.ref & RT_LEAF_BIT) ? -2.0f : box_area(r.b);
}

// One axis of a 64-byte node: base, step and the bytes of the children's
// planes.  The children's extent takes bytes 1 to 251; the step is at least
// 2^-19 of the coordinates, so that a plane's own rounding is below 0.04
// steps, and planes are moved outwards by 0.1 steps before they are rounded.
// A child with a NaN box gets an inside-out one, an axis beyond 1e23 a NaN
// base (every child passes).
__device__ __forceinline__ void quantize_axis(const float (&lo)[4], const float (&hi)[4], float &base, float &step,
                                              uint32_t &ql, uint32_t &qh) {
    const float l = fminf(fminf(lo[0], lo[1]), fminf(lo[2], lo[3])), h = fmaxf(fmaxf(hi[0], hi[1]), fmaxf(hi[2], hi[3]));
    ql = 0xffffffffu;
    qh = 0u;
    base = 0.0f;
    step = 1.0f;
    if (!(l == l)) return;  // no child has a box
    const float big = fmaxf(fabsf(l), fabsf(h)), s = fmaxf(fmaxf((h - l) * (1.0f / 248.0f), big * 1.9073486e-6f), 1e-30f);
    if (!(big < 1e23f)) {
        base = __int_as_float(0x7fc00000);
        return;
    }
    step = 32768.0f * s;
    base = (l - 2.0f * s) - step;
    const float zero = base + step, is = 1.0f / s;
    ql = qh = 0u;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const bool box = lo[c] == lo[c];
        const float a = floorf(fmaf(lo[c] - zero, is, -0.1f)), b = ceilf(fmaf(hi[c] - zero, is, 0.1f));
        ql |= (box ? (uint32_t)fminf(fmaxf(a, 0.0f), 255.0f) : 255u) << (8 * c);
        qh |= (box ? (uint32_t)fminf(fmaxf(b, 0.0f), 255.0f) : 0u) << (8 * c);
    }
}
__device__ __forceinline__ void store_qnode(float4 *q, const float (&lo)[3][4], const float (&hi)[3][4], float4 refs) {
    float base[3], step[3];
    uint32_t ql[3], qh[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) quantize_axis(lo[a], hi[a], base[a], step[a], ql[a], qh[a]);
    auto f = [](uint32_t u) { return __uint_as_float(u); };
    q[0] = make_float4(base[0], base[1], base[2], step[0]);
    q[1] = make_float4(step[1], step[2], f(ql[0]), f(qh[0]));
    q[2] = make_float4(f(ql[1]), f(qh[1]), f(ql[2]), f(qh[2]));
    q[3] = refs;
}

// The 4-wide tree.  The children of a wide node that starts from binary node
// e are found by greedy expansion (the internal child of largest surface area
// is replaced by its two children, twice), which depends on e's descendants
// alone; so every binary node is expanded as if it were the start of a wide
// node, all in one launch, and a wide node has the index of the binary node
// it starts from.  The nodes no other refers to (about half) are never read.
// Top-down, level by level, took 63 launches (276 us at 300k Gaussians, 181 us
// at 4k; 105 and 40 us with one block for the top and a thread per subtree).
__global__ void __launch_bounds__(128) k_wide(const float4 *__restrict__ nodes, int64_t ni, float4 *wide,
                                              float4 *qwide) {
    for (int64_t e = blockIdx.x * 128ll + threadIdx.x; e < ni; e += (int64_t)gridDim.x * 128) {
        // 2 children, then the larger's two behind the other, then the largest
        // of three replaced by the last and its two children appended
        WideSlot s0, s1, s2, s3;
        s2.ref = s3.ref = RT_EMPTY;
#pragma unroll
        for (int k = 0; k < 6; ++k) s2.b[k] = s3.b[k] = __int_as_float(0x7fc00000);
        wide_children(nodes, (int32_t)e, s0, s1);
        if (fmaxf(s0.area, s1.area) > -2.0f) {
            const bool first = !(s1.area > s0.area);
            const int32_t x = (int32_t)(first ? s0.ref : s1.ref);
            if (first) s0 = s1;
            wide_children(nodes, x, s1, s2);
            const float best = fmaxf(s0.area, fmaxf(s1.area, s2.area));
            if (best > -2.0f) {
                int32_t y;
                if (s0.area == best) {
                    y = (int32_t)s0.ref;
                    s0 = s2;
                } else if (s1.area == best) {
                    y = (int32_t)s1.ref;
                    s1 = s2;
                } else {
                    y = (int32_t)s2.ref;
                }
                wide_children(nodes, y, s2, s3);
            }
        }
        float4 *w = wide + 8 * e;
#pragma unroll
        for (int k = 0; k < 6; ++k) w[k] = make_float4(s0.b[k], s1.b[k], s2.b[k], s3.b[k]);
        const float4 refs = make_float4(__uint_as_float(s0.ref), __uint_as_float(s1.ref), __uint_as_float(s2.ref),
                                        __uint_as_float(s3.ref));
        w[6] = refs;
        w[7] = make_float4(0.f, 0.f, 0.f, 0.f);
        float lo[3][4], hi[3][4];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a][0] = s0.b[2 * a], lo[a][1] = s1.b[2 * a], lo[a][2] = s2.b[2 * a], lo[a][3] = s3.b[2 * a];
            hi[a][0] = s0.b[2 * a + 1], hi[a][1] = s1.b[2 * a + 1], hi[a][2] = s2.b[2 * a + 1];
            hi[a][3] = s3.b[2 * a + 1];
        }
        store_qnode(qwide + 4 * e, lo, hi, refs);
    }
}

// Refit of the 4-wide tree with its slots kept, after the binary tree's: the
// box of a child is the leaf's, or the union of the binary node's two.
// A thread per child, the four of a node side by side; lane a < 3 of them then
// quantizes axis a of the 64-byte node.
__global__ void __launch_bounds__(256) k_refit_wide(const float *__restrict__ leafbox, const float4 *__restrict__ nodes,
                                                    int64_t ni, float *wide, float *qwide) {
    const int64_t total = (4 * ni + 31) / 32 * 32;  // whole warps
    for (int64_t j = blockIdx.x * 256ll + threadIdx.x; j < total; j += (int64_t)gridDim.x * 256) {
        const bool in = j < 4 * ni;
        float *w = wide + 32 * (in ? j >> 2 : 0) + (j & 3);
        const uint32_t r = in ? __float_as_uint(w[24]) : RT_EMPTY;
        const float none = __int_as_float(0x7fc00000);
        float lo[3] = {none, none, none}, hi[3] = {none, none, none};
        if (r != RT_EMPTY) {
            if (r & RT_LEAF_BIT) {
                const float *b = leafbox + 6 * (int64_t)(r & ~RT_LEAF_BIT);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    lo[c] = b[c];
                    hi[c] = b[3 + c];
                }
            } else {
                const float4 x = nodes[4 * (int64_t)r], y = nodes[4 * (int64_t)r + 1], z = nodes[4 * (int64_t)r + 2];
                lo[0] = fminf(x.x, y.z); hi[0] = fmaxf(x.y, y.w);
                lo[1] = fminf(x.z, z.x); hi[1] = fmaxf(x.w, z.y);
                lo[2] = fminf(y.x, z.z); hi[2] = fmaxf(y.y, z.w);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                w[8 * c] = lo[c];
                w[8 * c + 4] = hi[c];
            }
        }
        const int axis = (int)(j & 3);
        float l4[4], h4[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float l = __shfl_sync(0xffffffffu, lo[c], k, 4), h = __shfl_sync(0xffffffffu, hi[c], k, 4);
                if (c == axis || c == 0) {
                    l4[k] = l;
                    h4[k] = h;
                }
            }
        if (!in || axis == 3) continue;
        float base, step;
        uint32_t ql, qh;
        quantize_axis(l4, h4, base, step, ql, qh);
        float *q = qwide + 16 * (j >> 2);
        q[axis] = base;
        q[3 + axis] = step;
        q[6 + 2 * axis] = __uint_as_float(ql);
        q[7 + 2 * axis] = __uint_as_float(qh);
    }
}

__global__ void k_export_boxes(const float4 *__restrict__ nodes, int64_t m, float *boxes,
                               int32_t *left, int32_t *right) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        float4 a = nodes[4 * i], b = nodes[4 * i + 1], c = nodes[4 * i + 2], r = nodes[4 * i + 3];
        if (boxes) {
            float *o = boxes + 12 * i;
            o[0] = a.x; o[1] = a.z; o[2] = b.x; o[3] = a.y; o[4] = a.w; o[5] = b.y;
            o[6] = b.z; o[7] = c.x; o[8] = c.z; o[9] = b.w; o[10] = c.y; o[11] = c.w;
        }
        if (left) left[i] = (int32_t)__float_as_uint(r.x);
        if (right) right[i] = (int32_t)__float_as_uint(r.y);
    }
}

// Keys per thread of a sort's tiles: small tiles until there are a few for
// every multiprocessor, larger ones beyond (fewer counts to scan).
int sort_items(int64_t n) { return n <= (int64_t(1) << 17) ? 4 : n <= (int64_t(1) << 19) ? 8 : 16; }
int sort_tiles(int64_t n) {
    const int64_t tile = (int64_t)kSortThreads * sort_items(n);
    return (int)((n + tile - 1) / tile);
}
template <int ITEMS>
void radix_pass(const uint32_t *k0, const int32_t *v0, int64_t n, int shift, int nblk, uint32_t *counts,
                uint32_t *k1, int32_t *v1, cudaStream_t st) {
    k_radix_hist<ITEMS><<<nblk, kSortThreads, 0, st>>>(k0, n, shift, nblk, counts);
    uint32_t *totals = counts + (int64_t)kRadix * nblk;
    k_radix_scan<<<kRadix, 256, 0, st>>>(counts, nblk, totals);
    k_radix_scatter<ITEMS><<<nblk, kSortThreads, 0, st>>>(k0, v0, n, shift, nblk, counts, totals, k1, v1);
}
// counts: kRadix * (sort_tiles(n) + 1) words.
// `passes` 8-bit passes from (k0, v0) to (k1, v1) and back, the arrays'
// names exchanged with each: the result is in (k0, v0).
void radix_sort(uint32_t *&k0, int32_t *&v0, uint32_t *&k1, int32_t *&v1, int64_t n, int passes, uint32_t *counts,
                cudaStream_t st) {
    const int nblk = sort_tiles(n), items = sort_items(n);
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = pass * kRadixBits;
        if (items == 4) radix_pass<4>(k0, v0, n, shift, nblk, counts, k1, v1, st);
        else if (items == 8) radix_pass<8>(k0, v0, n, shift, nblk, counts, k1, v1, st);
        else radix_pass<16>(k0, v0, n, shift, nblk, counts, k1, v1, st);
        uint32_t *tk = k0; k0 = k1; k1 = tk;
        int32_t *tv = v0; v0 = v1; v1 = tv;
    }
}

int grid_for(int64_t n, int threads) {
    int64_t g = (n + threads - 1) / threads;
    int64_t cap = (int64_t)rt_num_sms() * 16;
    if (g > cap) g = cap;
    return g < 1 ? 1 : (int)g;
}

int bounds_grid(int64_t n) {
    const int64_t g = (n + 511) / 512, cap = 2 * (int64_t)rt_num_sms();
    return (int)(g < 1 ? 1 : g < cap ? g : cap);
}
int refit_grid(int64_t n) {
    const int64_t g = (n + kRefitLeaves - 1) / kRefitLeaves, cap = 16 * (int64_t)rt_num_sms();
    return (int)(g < 1 ? 1 : g < cap ? g : cap);
}

void launch_refit(const float *leafbox, const int32_t *parent, int64_t n, float4 *nodes, uint32_t *arrivals,
                  uint32_t *levels, cudaStream_t st) {
    if (n > 8 * kRefitLeaves) {
        k_refit<false><<<refit_grid(n), kRefitLeaves, 0, st>>>(leafbox, parent, n, nodes, arrivals, levels);
        return;
    }
    int blocks = 1;  // a power of two: every cluster size of up to 8 is portable
    while (blocks * kRefitLeaves < n) blocks *= 2;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kRefitLeaves);
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)blocks;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_refit<true>, leafbox, parent, n, nodes, arrivals, levels);  // rt_check_launch reports
}

float host_ord2f(uint32_t u) {
    u = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
    float f;
    memcpy(&f, &u, sizeof(f));
    return f;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

rt_status rt_sort_pairs_u32(uint32_t *keys, int32_t *vals, int64_t n, int bits, rt_stream_t stream) {
    if (n <= 1 || bits <= 0) return RT_OK;
    if (n > (int64_t(1) << 31)) return RT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int nblk = sort_tiles(n);
    auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t bk = up(size_t(n) * 4), bc = up(size_t(kRadix) * (nblk + 1) * 4);
    void *blk = nullptr;
    RT_TRY(rt_alloc(&blk, 2 * bk + bc, stream));
    uint32_t *k0 = keys, *k1 = (uint32_t *)blk, *counts = (uint32_t *)((char *)blk + 2 * bk);
    int32_t *v0 = vals, *v1 = (int32_t *)((char *)blk + bk);
    const int passes = bits >= 32 ? 4 : (bits + kRadixBits - 1) / kRadixBits;
    radix_sort(k0, v0, k1, v1, n, passes, counts, st);
    rt_status r = rt_check_launch();
    if (r == RT_OK && k0 != keys &&
        (cudaMemcpyAsync(keys, k0, size_t(n) * 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
         cudaMemcpyAsync(vals, v0, size_t(n) * 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess)) {
        cudaGetLastError();
        r = RT_ERR_CUDA;
    }
    rt_free(blk, stream);
    return r;
}

extern "C" rt_status rt_build_bvh(const float *mean, const float *scale, const float *quat,
                                  const float *opacity, int64_t n, const rt_params *params,
                                  rt_stream_t stream, rt_bvh **out) {
    if (!out) return RT_ERR_INVALID_ARG;
    *out = nullptr;
    if (n < 0 || n >= (int64_t)0x7fffffff) return RT_ERR_INVALID_ARG;
    if (n > 0 && (!mean || !scale || !quat || !opacity)) return RT_ERR_INVALID_ARG;
    rt_params prm;
    rt_params_default(&prm);
    if (params) prm = *params;
    if (!(prm.k_sigma > 0.f) || !(prm.alpha_min > 0.f && prm.alpha_min < 1.f) ||
        !(prm.t_min >= 0.f && prm.t_min < 1.f) || !(prm.origin_eps >= 0.f) ||
        (prm.box_mode != 0 && prm.box_mode != 1) || (prm.deterministic != 0 && prm.deterministic != 1))
        return RT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;

    rt_bvh *b = new rt_bvh();
    b->n = n;
    b->params = prm;
    const int64_t ni = n > 1 ? n - 1 : 0;
    size_t off_g = 0;
    size_t off_nd = off_g + align256(sizeof(float4) * 4 * (size_t)n);
    size_t off_perm = off_nd + align256(sizeof(float4) * 4 * (size_t)ni);
    size_t off_rank = off_perm + align256(sizeof(int32_t) * (size_t)n);
    size_t off_keys = off_rank + align256(sizeof(int32_t) * (size_t)n);
    size_t off_par = off_keys + align256(sizeof(uint64_t) * (size_t)n);
    size_t off_bnd = off_par + align256(sizeof(int32_t) * (size_t)(n > 0 ? 2 * n - 1 : 0));
    size_t off_grp = off_bnd + 256;
    size_t off_wide = off_grp + align256(sizeof(int2) * (size_t)n);
    size_t off_qwide = off_wide + align256(sizeof(float4) * 8 * (size_t)ni);
    size_t total = off_qwide + align256(sizeof(float4) * 4 * (size_t)ni);
    rt_status s = rt_alloc(&b->block, total, stream);
    if (s != RT_OK) {
        delete b;
        return s;
    }
    char *base = (char *)b->block;
    b->bytes = (int64_t)total;
    b->gauss = (float4 *)(base + off_g);
    b->nodes = (float4 *)(base + off_nd);
    b->perm = (int32_t *)(base + off_perm);
    b->rank = (int32_t *)(base + off_rank);
    b->keys = (uint64_t *)(base + off_keys);
    b->parent = (int32_t *)(base + off_par);
    b->bounds = (float *)(base + off_bnd);
    b->groups = (int2 *)(base + off_grp);
    b->n_groups = 0;
    b->wide = (float4 *)(base + off_wide);
    b->qwide = (float4 *)(base + off_qwide);
    b->n_wide = 0;
    b->levels = 0;
    for (int c = 0; c < 3; ++c) b->lo[c] = b->hi[c] = 0.f;
    if (n == 0) {
        *out = b;
        return RT_OK;
    }

    // scratch: scene words | codes, vals x2 | counts | leafbox | arrivals
    const bool small = n <= kSmallSort;
    const int64_t mc = small ? 0 : (int64_t)kRadix * (sort_tiles(n) + 1);
    size_t s_k0 = SCN_BYTES;
    size_t s_v0 = s_k0 + align256(4 * (size_t)n);
    size_t s_k1 = s_v0 + align256(4 * (size_t)n);
    size_t s_v1 = s_k1 + align256(4 * (size_t)n);
    size_t s_cnt = s_v1 + align256(4 * (size_t)n);
    size_t s_leaf = s_cnt + align256(4 * (size_t)mc);
    size_t s_arr = s_leaf + align256(24 * (size_t)n);
    size_t s_total = s_arr + align256(4 * (size_t)ni);
    void *scratch = nullptr;
    s = rt_alloc(&scratch, s_total, stream);
    if (s != RT_OK) {
        rt_free(b->block, stream);
        delete b;
        return s;
    }
    char *sb = (char *)scratch;
    uint32_t *scn = (uint32_t *)sb;
    uint32_t *k0 = (uint32_t *)(sb + s_k0), *k1 = (uint32_t *)(sb + s_k1);
    int32_t *v0 = (int32_t *)(sb + s_v0), *v1 = (int32_t *)(sb + s_v1);
    uint32_t *counts = (uint32_t *)(sb + s_cnt);
    float *leafbox = (float *)(sb + s_leaf);
    uint32_t *arrivals = (uint32_t *)(sb + s_arr);

    rt_status result = RT_OK;
    uint32_t res[SCN_WORDS] = {0};  // host copy of the scene words
    if (cudaMemsetAsync(scn, 0, SCN_BYTES, st) != cudaSuccess) result = RT_ERR_CUDA;
    if (result == RT_OK) {
        k_bounds<<<bounds_grid(n), 512, 0, st>>>(mean, scale, quat, opacity, n, scn);
        if (small) {
            k_sort_small<<<((int)n + 31) / 32, 1024, 0, st>>>(mean, (int)n, scn, b->bounds, k0, v0);
        } else {
            k_morton<<<grid_for(n, 256), 256, 0, st>>>(mean, n, scn, b->bounds, k0, v0);
            radix_sort(k0, v0, k1, v1, n, 4, counts, st);
        }
        k_prep<<<grid_for(n, 128), 128, 0, st>>>(mean, scale, quat, opacity, v0, k0, n, prm, scn, b->gauss, leafbox,
                                                 b->perm, b->rank, b->keys);
        const int kb = grid_for(ni, 128), gb = grid_for((n + 63) / 64, 4);
        k_topology<<<kb + gb, 128, 0, st>>>(b->keys, n, b->nodes, b->parent, arrivals, kb, b->gauss, leafbox, b->groups,
                                            scn + SCN_GROUPS);
        if (n == 1) {
            if (cudaMemsetAsync(b->parent, 0xff, sizeof(int32_t), st) != cudaSuccess) result = RT_ERR_CUDA;  // -1
        } else {
            launch_refit(leafbox, b->parent, n, b->nodes, arrivals, scn + SCN_LEVELS, st);
            k_wide<<<grid_for(ni, 128), 128, 0, st>>>(b->nodes, ni, b->wide, b->qwide);
            b->n_wide = ni;
        }
        if (rt_check_launch() != RT_OK) result = RT_ERR_CUDA;
    }
    if (result == RT_OK && (cudaMemcpyAsync(res, scn, sizeof(res), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                            cudaStreamSynchronize(st) != cudaSuccess))
        result = RT_ERR_CUDA;
    rt_free(scratch, stream);
    if (result == RT_OK && res[SCN_BAD]) result = RT_ERR_INVALID_ARG;
    if (result != RT_OK) {
        rt_free(b->block, stream);
        delete b;
        return result;
    }
    for (int c = 0; c < 3; ++c) {
        b->lo[c] = host_ord2f(~res[c]);
        b->hi[c] = host_ord2f(res[3 + c]);
    }
    b->n_groups = res[SCN_GROUPS];
    b->levels = (int32_t)res[SCN_LEVELS];
    *out = b;
    return RT_OK;
}

extern "C" rt_status rt_bvh_refit(rt_bvh *b, const float *mean, const float *scale, const float *quat,
                                  const float *opacity, rt_stream_t stream) {
    if (!b) return RT_ERR_INVALID_ARG;
    const int64_t n = b->n;
    if (n == 0) return RT_OK;
    if (!mean || !scale || !quat || !opacity) return RT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t ni = n > 1 ? n - 1 : 0;
    // scratch: scene words | leaf boxes | binary arrivals
    const size_t s_leaf = SCN_BYTES, s_arr = s_leaf + align256(24 * (size_t)n);
    void *scratch = nullptr;
    RT_TRY(rt_alloc(&scratch, s_arr + align256(4 * (size_t)ni) + 256, stream));
    char *sb = (char *)scratch;
    uint32_t *scn = (uint32_t *)sb;
    float *leafbox = (float *)(sb + s_leaf);
    uint32_t *arrivals = (uint32_t *)(sb + s_arr);
    rt_status result = RT_OK;
    do {
        if (cudaMemsetAsync(scn, 0, SCN_BYTES, st) != cudaSuccess) {
            result = RT_ERR_CUDA;
            break;
        }
        k_bounds<<<bounds_grid(n), 512, 0, st>>>(mean, scale, quat, opacity, n, scn);
        k_report_invalid<<<1, 1, 0, st>>>(scn + SCN_BAD, rt_status_ptr());
        k_prep<<<grid_for(n, 128), 128, 0, st>>>(mean, scale, quat, opacity, b->perm, nullptr, n, b->params, scn,
                                                 b->gauss, leafbox, nullptr, nullptr, nullptr);
        if (n > 1) {
            if (cudaMemsetAsync(arrivals, 0, 4 * (size_t)ni, st) != cudaSuccess) {
                result = RT_ERR_CUDA;
                break;
            }
            launch_refit(leafbox, b->parent, n, b->nodes, arrivals, scn + SCN_LEVELS, st);
        }
        if (b->n_wide > 0)
            k_refit_wide<<<grid_for(4 * ni, 256), 256, 0, st>>>(leafbox, b->nodes, ni, (float *)b->wide,
                                                                       (float *)b->qwide);
        result = rt_check_launch();
    } while (0);
    rt_free(scratch, stream);
    return result;
}

extern "C" rt_status rt_bvh_destroy(rt_bvh *bvh, rt_stream_t stream) {
    if (!bvh) return RT_ERR_INVALID_ARG;
    rt_free(bvh->block, stream);
    delete bvh;
    return RT_OK;
}

extern "C" rt_status rt_bvh_info(const rt_bvh *bvh, int64_t *n, float *lo, float *hi, int64_t *bytes) {
    if (!bvh) return RT_ERR_INVALID_ARG;
    if (n) *n = bvh->n;
    for (int c = 0; c < 3; ++c) {
        if (lo) lo[c] = bvh->lo[c];
        if (hi) hi[c] = bvh->hi[c];
    }
    if (bytes) *bytes = bvh->bytes;
    return RT_OK;
}

extern "C" rt_status rt_bvh_export(const rt_bvh *bvh, uint64_t *keys, int32_t *left, int32_t *right,
                                   int32_t *parent, float *boxes, rt_stream_t stream) {
    if (!bvh) return RT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    int64_t n = bvh->n;
    if (n == 0) return RT_OK;
    if (keys && cudaMemcpyAsync(keys, bvh->keys, 8 * (size_t)n, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return RT_ERR_CUDA;
    if (parent && cudaMemcpyAsync(parent, bvh->parent, 4 * (size_t)(2 * n - 1), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return RT_ERR_CUDA;
    if (n > 1 && (boxes || left || right)) {
        k_export_boxes<<<grid_for(n - 1, 256), 256, 0, st>>>(bvh->nodes, n - 1, boxes, left, right);
        return rt_check_launch();
    }
    return RT_OK;
}
