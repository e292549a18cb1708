// rt_shade.cu -- consumers of the visibility: the per-Gaussian PBR colour of
// Eq. 10 (Sec. 3.3) and ambient occlusion.
//
// Sec. 3.3 computes a PBR colour per Gaussian by summing the rendering
// equation over N_s hemisphere directions about the Gaussian's normal, with
// the incident light of Eq. 8 (visibility x a global environment map plus
// per-Gaussian SH indirect light) and the simplified Disney BRDF of Eq. 9;
// Sec. 4.2 precomputes the visibility of those directions.  Two forms:
//   - from a visibility table V[n, K] (the paper's order: precompute once,
//     shade every iteration): one or several threads per Gaussian;
//   - fused: one warp per 32 Morton-adjacent Gaussians traces all K rays of
//     each and shades in the epilogue, so V is never written.
// Ambient occlusion is the fused form with the mean of T as the epilogue.
// Both forms share the map lookup and the BRDF term; the SH light is summed in
// the Gaussian's frame by the first and in the world's by the second (the same
// value up to rounding).
#include <string.h>

#include "rt_shaft.cuh"

namespace {

constexpr int kMaxEnvTexels = 2048;  // map staged in shared memory, 16 bytes a texel (32 KB)
constexpr float kPi = 3.14159265358979f;
constexpr float kF0 = 0.04f;
constexpr float kRoughMin = 0.04f;
// Default traversal of hemisphere sets in the fused kernels: one thread per
// ray over the 4-wide tree (measured faster than the warp packet on the 2M
// object scene, where the lanes' k-th directions differ with the normals).
constexpr int kHemiStrat = 4;

struct ShadeDev {
    const float *albedo, *rough, *sh, *env;
    const float *normals, *hemi;
    int32_t env_h, env_w, K;
    float vh, uw;  // env_h / pi, env_w / (2 pi)
    float3 cam;
};

__device__ __forceinline__ float dot3f(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

// atan2(y, x) for (y, x) != 0: atan of the smaller over the larger magnitude
// by a polynomial (minimax fit, Remez exchange, of atan(t) on [0, 1] with
// weight 1: degree 17, absolute error 8e-8 in float32, as CUDA's atan2f),
// then the octant; 20 instructions.
__device__ __forceinline__ float atan2_poly(float y, float x) {
    const float ax = fabsf(x), ay = fabsf(y);
    const float t = __fdividef(fminf(ax, ay), fmaxf(ax, ay)), s = t * t;
    float p = 0.0024566669f;
    p = fmaf(p, s, -0.0144011294f);
    p = fmaf(p, s, 0.0397808552f);
    p = fmaf(p, s, -0.0723482594f);
    p = fmaf(p, s, 0.104989313f);
    p = fmaf(p, s, -0.141612247f);
    p = fmaf(p, s, 0.199859068f);
    p = fmaf(p, s, -0.333325982f);
    p = fmaf(p, s, 0.999999881f);
    float r = p * t;
    r = ay > ax ? 0.5f * kPi - r : r;
    r = x < 0.0f ? kPi - r : r;
    return copysignf(r, y);
}

// Bilinear lookup between pixel centres of the equirectangular map (row i:
// polar angles [i pi/h, (i+1) pi/h]; azimuth wraps, polar angle clamps).
// env: one texel per float4; vh = h / pi, uw = w / (2 pi).  The polar angle
// comes from both legs (acos alone loses half the digits at the poles).
__device__ __forceinline__ void env_lookup(const float4 *env, int h, int w, float vh, float uw, float3 d,
                                           float L[3]) {
    const float r2 = fmaf(d.x, d.x, d.y * d.y);
    const float v = fmaf(atan2_poly(__fsqrt_rn(r2), d.z), vh, -0.5f);
    const float ph = r2 > 0.0f ? atan2_poly(d.y, d.x) : 0.0f;
    const float u = fmaf(ph, uw, ph < 0.0f ? (float)w - 0.5f : -0.5f);
    const float fv = floorf(v), fu = floorf(u);
    const float bv = v - fv, bu = u - fu;
    const int i = min(max((int)fv, -1), h - 1), j = min(max((int)fu, -1), w - 1);
    const int i0 = max(i, 0) * w, i1 = min(i + 1, h - 1) * w;
    const int j0 = j < 0 ? w - 1 : j, j1 = j + 1 == w ? 0 : j + 1;
    const float4 e00 = env[i0 + j0], e01 = env[i0 + j1], e10 = env[i1 + j0], e11 = env[i1 + j1];
    auto mix = [&](float a00, float a01, float a10, float a11) {
        const float a = fmaf(bu, a01 - a00, a00), b = fmaf(bu, a11 - a10, a10);
        return fmaf(bv, b - a, a);
    };
    L[0] = mix(e00.x, e01.x, e10.x, e11.x);
    L[1] = mix(e00.y, e01.y, e10.y, e11.y);
    L[2] = mix(e00.z, e01.z, e10.z, e11.z);
}

// Per-Gaussian constants of the shading sum: normal and view direction, and
// of Eq. 9's D F G / (4 (n.wi)(n.wo)) with GGX D (alpha = r^2), Schlick F
// (F0 = 0.04) and Smith-Schlick G (k = (r+1)^2/8), G1(x)/x = 1/(x(1-k)+k)
// so that it stays finite at grazing angles, what does not depend on wi.
struct ShadeLane {
    float3 n, wo;
    float a2, k, cs;  // alpha^2, k, alpha^2 / (4 pi (n.wo (1-k) + k))
    float3 alb;       // albedo / pi
};

__device__ __forceinline__ ShadeLane shade_lane(const ShadeDev &S, const HemiFrame &f, int64_t g, float4 mu) {
    ShadeLane L;
    L.n = f.n;
    float3 wo = make_float3(S.cam.x - mu.x, S.cam.y - mu.y, S.cam.z - mu.z);
    const float il = rsqrtf(dot3f(wo, wo));
    L.wo = make_float3(wo.x * il, wo.y * il, wo.z * il);
    L.alb = make_float3(__ldg(S.albedo + 3 * g) * (1.0f / kPi), __ldg(S.albedo + 3 * g + 1) * (1.0f / kPi),
                        __ldg(S.albedo + 3 * g + 2) * (1.0f / kPi));
    const float r = fminf(fmaxf(__ldg(S.rough + g), kRoughMin), 1.0f);
    const float al = r * r;
    L.a2 = al * al;
    L.k = (r + 1.0f) * (r + 1.0f) * 0.125f;
    L.cs = L.a2 / (4.0f * kPi * fmaf(fmaxf(dot3f(f.n, L.wo), 0.0f), 1.0f - L.k, L.k));
    return L;
}

// Specular term; nl = max(n.wi, 0).  The GGX denominator 1 + (n.h)^2
// (alpha^2 - 1) is evaluated as |n x h|^2 + (n.h)^2 alpha^2, which has no
// cancellation near the mirror direction.  (At alpha^2 = 2.6e-6 the rounding
// of h still moves it by 1e-4 of itself there; written in the Gaussian's
// frame it is 7 % faster and no less accurate, but rounds differently.)
__device__ __forceinline__ float spec_term(const ShadeLane &L, float3 wi, float nl) {
    const float3 hv = make_float3(wi.x + L.wo.x, wi.y + L.wo.y, wi.z + L.wo.z);
    const float hl2 = dot3f(hv, hv);
    if (!(hl2 > 0.0f)) return 0.0f;
    const float inv = rsqrtf(hl2);
    const float3 n = L.n, h = make_float3(hv.x * inv, hv.y * inv, hv.z * inv);
    const float nh = dot3f(n, h), vh = fmaxf(dot3f(L.wo, h), 0.0f);
    const float3 cr = make_float3(n.y * h.z - n.z * h.y, n.z * h.x - n.x * h.z, n.x * h.y - n.y * h.x);
    const float q = dot3f(cr, cr) + nh * nh * L.a2;
    const float m = 1.0f - vh, m2 = m * m;
    const float F = kF0 + (1.0f - kF0) * (m2 * m2 * m);
    return __fdividef(L.cs * F, q * q * fmaf(nl, 1.0f - L.k, L.k));
}

// One term of Eq. 10: acc += (b/pi + f_s) (V L_direct + max(0, SH)) max(n.wi, 0)
// for the direction wi with n.wi = hz; Li: the SH light.
__device__ __forceinline__ void shade_add(const ShadeDev &S, const float4 *env, const ShadeLane &L, float3 wi,
                                          float hz, float V, const float (&Li)[3], float acc[3]) {
    const float nl = fmaxf(hz, 0.0f);
    const float fs = spec_term(L, wi, nl);
    float Ld[3];
    env_lookup(env, S.env_h, S.env_w, S.vh, S.uw, wi, Ld);
    const float alb[3] = {L.alb.x, L.alb.y, L.alb.z};
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[c] = fmaf((alb[c] + fs) * nl, fmaf(V, Ld[c], Li[c]), acc[c]);
}

constexpr float kSh0 = 0.282094791773878f, kSh1 = 0.488602511902920f, kSh2a = 1.092548430592079f,
                kSh2b = 0.315391565252520f, kSh2c = 0.546274215296040f;

// max(0, SH light) of Gaussian g (27 coefficients) along the world direction.
__device__ __forceinline__ void sh_light(const float *sh, float3 wi, float (&Li)[3]) {
    const float x = wi.x, y = wi.y, z = wi.z;
    const float Y[9] = {kSh0, -kSh1 * y, kSh1 * z, -kSh1 * x, kSh2a * x * y, -kSh2a * y * z,
                        kSh2b * (2.0f * z * z - x * x - y * y), -kSh2a * x * z, kSh2c * (x * x - y * y)};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float s = 0.0f;
#pragma unroll
        for (int j = 0; j < 9; ++j) s += __ldg(sh + 3 * j + c) * Y[j];
        Li[c] = fmaxf(s, 0.0f);
    }
}

__device__ __forceinline__ void load_env(const ShadeDev &S, float4 *env_s) {
    for (int i = threadIdx.x; i < S.env_h * S.env_w; i += blockDim.x)
        env_s[i] = make_float4(__ldg(S.env + 3 * i), __ldg(S.env + 3 * i + 1), __ldg(S.env + 3 * i + 2), 0.0f);
    __syncthreads();
}

// The SH light of one channel as a quadratic form in the local direction h:
// q[0] + q[1..3] . h + q[4] (hx^2 - hz^2) + q[5] (hy^2 - hz^2) + q[6] hx hy +
// q[7] hx hz + q[8] hy hz (the form is traceless).
__device__ __forceinline__ void sh_local(const float *sh, int c, const HemiFrame &f, float (&q)[9]) {
    float s[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) s[j] = __ldg(sh + 3 * j + c);
    const float3 b = make_float3(-kSh1 * s[3], -kSh1 * s[1], kSh1 * s[2]);
    const float xx = fmaf(kSh2c, s[8], -kSh2b * s[6]), yy = fmaf(-kSh2c, s[8], -kSh2b * s[6]), zz = 2.0f * kSh2b * s[6];
    const float xy = 0.5f * kSh2a * s[4], yz = -0.5f * kSh2a * s[5], xz = -0.5f * kSh2a * s[7];
    auto mul = [&](float3 v) {
        return make_float3(fmaf(xx, v.x, fmaf(xy, v.y, xz * v.z)), fmaf(xy, v.x, fmaf(yy, v.y, yz * v.z)),
                           fmaf(xz, v.x, fmaf(yz, v.y, zz * v.z)));
    };
    const float3 m1 = mul(f.t1), m2 = mul(f.t2), mn = mul(f.n);
    q[0] = kSh0 * s[0];
    q[1] = dot3(b, f.t1);
    q[2] = dot3(b, f.t2);
    q[3] = dot3(b, f.n);
    q[4] = dot3(f.t1, m1);
    q[5] = dot3(f.t2, m2);
    q[6] = 2.0f * dot3(f.t1, m2);
    q[7] = 2.0f * dot3(f.t1, mn);
    q[8] = 2.0f * dot3(f.t2, mn);
}

// Shading from a visibility table: LANES threads per Gaussian (original
// order), each a share of its K terms.  What a term needs of its direction in
// the Gaussian's frame is the same for every Gaussian, so it is tabulated once
// per block: the direction and the five quadratic monomials of the SH light,
// whose 27 coefficients each thread turns into its frame once and keeps in
// registers, as it does the constants of the BRDF.  The direction itself is
// turned into the world only for the map lookup.
// Bound: instruction issue (1M x 64 terms: 0.50 ms, 1.74 ms when each term
// loaded the 27 coefficients anew, from 27 x 32 different lines a warp, and
// called acosf, atan2f and three integer remainders; the table's 4 bytes a
// term are 8 % of the memory's rate).  VEC: V is read four terms at a time.
constexpr int kShadeChunk = 128;  // tabulated directions
template <int LANES, bool SH, bool VEC>
__global__ void __launch_bounds__(128) k_pbr_shade_v(BvhDev b, ShadeDev S, const float *__restrict__ V,
                                                     float *__restrict__ rgb) {
    extern __shared__ float4 env_s[];  // env_h * env_w texels, then 2 per direction
    float4 *tab = env_s + S.env_h * S.env_w;
    load_env(S, env_s);
    const int sub = threadIdx.x & (LANES - 1);
    constexpr int per = 128 / LANES;  // Gaussians of a block
    const int64_t tiles = (b.n + per - 1) / per;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t g = tile * per + threadIdx.x / LANES;
        const bool valid = g < b.n;
        HemiFrame f;
        ShadeLane L;
        float q[3][9];
        if (valid) {
            f = hemi_frame(S.normals + 3 * g);
            L = shade_lane(S, f, g, __ldg(b.gauss + 4 * (int64_t)b.rank[g]));
            if (SH)
#pragma unroll
                for (int c = 0; c < 3; ++c) sh_local(S.sh + 27 * g, c, f, q[c]);
        }
        float acc[3] = {0.0f, 0.0f, 0.0f};
        for (int k0 = 0; k0 < S.K; k0 += kShadeChunk) {
            const int kn = min(kShadeChunk, S.K - k0);
            if (S.K > kShadeChunk || tile == blockIdx.x) {
                __syncthreads();
                for (int i = threadIdx.x; i < kn; i += 128) {
                    const float *h = S.hemi + 3 * (k0 + i);
                    const float x = __ldg(h), y = __ldg(h + 1), z = __ldg(h + 2);
                    tab[2 * i] = make_float4(x, y, z, x * y);
                    tab[2 * i + 1] = make_float4(x * x - z * z, y * y - z * z, x * z, y * z);
                }
                __syncthreads();
            }
            if (!valid) continue;
            const float *Vg = V + g * S.K + k0;
            auto term = [&](int k, float v) {
                const float4 h = tab[2 * k], m = tab[2 * k + 1];
                const float3 wi = hemi_rotate(f, h.x, h.y, h.z);
                float Li[3] = {0.0f, 0.0f, 0.0f};
                if (SH)
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        float s = fmaf(q[c][1], h.x, fmaf(q[c][2], h.y, fmaf(q[c][3], h.z, q[c][0])));
                        s = fmaf(q[c][4], m.x, fmaf(q[c][5], m.y, s));
                        s = fmaf(q[c][6], h.w, fmaf(q[c][7], m.z, fmaf(q[c][8], m.w, s)));
                        Li[c] = fmaxf(s, 0.0f);
                    }
                shade_add(S, env_s, L, wi, h.z, v, Li, acc);
            };
            if (VEC) {
                for (int k = 4 * sub; k < kn; k += 4 * LANES) {
                    const float4 v = __ldg(reinterpret_cast<const float4 *>(Vg + k));
                    term(k, v.x);
                    term(k + 1, v.y);
                    term(k + 2, v.z);
                    term(k + 3, v.w);
                }
            } else {
                for (int k = sub; k < kn; k += LANES) term(k, __ldg(Vg + k));
            }
        }
#pragma unroll
        for (int off = LANES / 2; off > 0; off >>= 1)
#pragma unroll
            for (int c = 0; c < 3; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], off);
        if (valid && sub == 0) {
            const float w = 2.0f * kPi / (float)S.K;
            rgb[3 * g] = acc[0] * w;
            rgb[3 * g + 1] = acc[1] * w;
            rgb[3 * g + 2] = acc[2] * w;
        }
    }
}

// Fused trace + reduction over all K rays of each Gaussian.  An item is a
// tile of 32 Morton-adjacent Gaussians; the warp traces ray k of all 32
// lanes together (STRAT 2: warp packet over the 4-wide tree; 4: one thread per
// ray) for k = 0..K-1.
// MODE 0: PBR colour (Eq. 10); MODE 1: ambient occlusion (mean of T).
template <int STRAT, int MODE>
__global__ void __launch_bounds__(128, 8) k_trace_reduce(BvhDev b, RaySetDev rs, ShadeDev S, float *__restrict__ out,
                                                         int *status, unsigned long long *work) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    __shared__ int2 stk_all[STRAT == 2 ? 4 * RT_WIDE_STACK : 1];
    int2 *stk = stk_all + (STRAT == 2 ? (threadIdx.x >> 5) * RT_WIDE_STACK : 0);
    extern __shared__ float4 env_s[];
    if (MODE == 0) load_env(S, env_s);
    const int64_t n_tiles = (b.n + 31) / 32;
    WorkCounts wc = {0, 0, 0};
    LaneLog lg;
    lg.ids = nullptr;
    lg.cap = 0;
    lg.count = 0;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(work, 1ull);
        item = __shfl_sync(FULL, item, 0);
        if ((int64_t)item >= n_tiles) break;
        const int64_t p = (int64_t)item * 32 + lane;
        const bool valid = p < b.n;
        float4 mu = make_float4(0.f, 0.f, 0.f, 0.f);
        int64_t g = 0;
        if (valid) {
            mu = __ldg(b.gauss + 4 * p);
            g = __float_as_int(__ldg(b.gauss + 4 * p + 1).w);
        }
        float acc[3] = {0.0f, 0.0f, 0.0f};
        for (int32_t k = 0; k < rs.K; ++k) {
            float3 o = make_float3(0.f, 0.f, 0.f), d = make_float3(0.f, 0.f, 1.f);
            if (valid) implicit_ray(rs, g * rs.K + k, k, g, mu, o, d);
            const int32_t src = valid ? (int32_t)p : -1;
            float T;
            if (STRAT == 4) T = valid ? trace_ray_wide<false>(b, o, d, src, lg, wc, status, far_first(rs)) : 1.0f;
            else T = trace_wide<false>(b, o, d, src, valid, lg, wc, status, stk);
            if (!valid) continue;
            if (MODE == 0) {
                // the per-Gaussian constants are rebuilt after each traversal
                // (a few dozen instructions and L1 hits) so that they hold no
                // registers across it
                const float4 m2 = __ldg(b.gauss + 4 * p);
                float Li[3] = {0.0f, 0.0f, 0.0f};
                if (S.sh) sh_light(S.sh + 27 * g, d, Li);
                shade_add(S, env_s, shade_lane(S, hemi_frame(S.normals + 3 * g), g, m2), d, __ldg(S.hemi + 3 * k + 2),
                          T, Li, acc);
            } else {
                acc[0] += T;
            }
        }
        if (!valid) continue;
        if (MODE == 0) {
            const float w = 2.0f * kPi / (float)rs.K;
            out[3 * g] = acc[0] * w;
            out[3 * g + 1] = acc[1] * w;
            out[3 * g + 2] = acc[2] * w;
        } else {
            out[g] = acc[0] / (float)rs.K;
        }
    }
}

// Ambient occlusion of a direction set: an item is a shaft group, traced
// along the K directions in turn, each lane summing its (up to two) rays.
__global__ void __launch_bounds__(128, kShaftBlocks) k_shaft_ao(BvhDev b, RaySetDev rs, int64_t n_groups,
                                                                       float *__restrict__ ao, int *status,
                                                                       unsigned long long *work) {
    __shared__ ShaftSmem<false> sm_all[4];
    ShaftSmem<false> &sm = sm_all[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(work, 1ull);
        item = __shfl_sync(0xffffffffu, item, 0);
        if ((int64_t)item >= n_groups) break;
        const int2 gr = __ldg(b.groups + item);
        float acc[2] = {0.0f, 0.0f};
        for (int32_t k = 0; k < rs.K; ++k) {
            shaft_group<false>(b, rs.eps, make_float3(__ldg(rs.dirs + 3 * k), __ldg(rs.dirs + 3 * k + 1), __ldg(rs.dirs + 3 * k + 2)),
                        gr.x, gr.y, status, sm);
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (lane + 32 * r < gr.y) {
                    const float T = sm.ro[lane + 32 * r].w;
                    acc[r] += T < b.t_min ? 0.0f : T;
                }
            __syncwarp();
        }
#pragma unroll
        for (int r = 0; r < 2; ++r)
            if (lane + 32 * r < gr.y)
                ao[__float_as_int(__ldg(b.gauss + 4 * (int64_t)(gr.x + lane + 32 * r) + 1).w)] = acc[r] / (float)rs.K;
    }
}

int grid_for(const void *kernel, int threads, size_t smem) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    return per_sm * rt_num_sms();
}

rt_status shade_dev(const rt_bvh *bvh, const rt_rayspec *rays, const rt_pbr_inputs *in, RaySetDev *rs,
                    ShadeDev *S) {
    if (!bvh || !rays || !in || rays->kind != RT_RAYS_HEMI || rays->ray_ids) return RT_ERR_INVALID_ARG;
    int64_t count = 0;
    RT_TRY(rt_rayset_dev(bvh, rays, rs, &count));
    if (in->env_h <= 0 || in->env_w <= 0 || (int64_t)in->env_h * in->env_w > kMaxEnvTexels || !in->env)
        return RT_ERR_INVALID_ARG;
    if (bvh->n > 0 && (!in->albedo || !in->roughness)) return RT_ERR_INVALID_ARG;
    memset(S, 0, sizeof(*S));
    S->albedo = in->albedo;
    S->rough = in->roughness;
    S->sh = in->sh;
    S->env = in->env;
    S->env_h = in->env_h;
    S->env_w = in->env_w;
    S->vh = (float)(in->env_h / 3.14159265358979323846);
    S->uw = (float)(in->env_w / 6.28318530717958647692);
    S->normals = rays->normals;
    S->hemi = rays->dirs;
    S->K = rays->n_dirs;
    S->cam = make_float3(in->cam[0], in->cam[1], in->cam[2]);
    return RT_OK;
}

// strat: 2 warp packet (per-lane directions), 3 shaft packet (DIRS, MODE 1),
// 4 one thread per ray; all over the 4-wide tree.
template <int MODE>
rt_status launch_reduce(const rt_bvh *bvh, const RaySetDev &rs, const ShadeDev &S, float *out, size_t smem,
                        int strat, cudaStream_t st) {
    unsigned long long *work = nullptr;
    RT_TRY(rt_alloc((void **)&work, sizeof(unsigned long long), st));
    rt_status res = RT_OK;
    if (cudaMemsetAsync(work, 0, sizeof(unsigned long long), st) != cudaSuccess) res = RT_ERR_CUDA;
    const BvhDev b = bvh_dev(bvh);
    if (res == RT_OK) {
#define RT_REDUCE(ST)                                                                     \
    do {                                                                                  \
        const int grid = grid_for((const void *)k_trace_reduce<ST, MODE>, 128, smem);     \
        k_trace_reduce<ST, MODE><<<grid, 128, smem, st>>>(b, rs, S, out, rt_status_ptr(), work); \
        res = rt_check_launch();                                                          \
    } while (0)
        // a tree of fewer than 2 Gaussians has no 4-wide form: strategy 4
        // handles it without touching one
        if (b.wide == nullptr && b.n >= 2) res = RT_ERR_UNSUPPORTED;
        else if (b.wide == nullptr) RT_REDUCE(4);
        else if (strat == 3) {  // ambient occlusion of a direction set
            const int grid = grid_for((const void *)k_shaft_ao, 128, 0);
            k_shaft_ao<<<grid, 128, 0, st>>>(b, rs, bvh->n_groups, out, rt_status_ptr(), work);
            res = rt_check_launch();
        }
        else if (strat == 2) RT_REDUCE(2);
        else RT_REDUCE(4);
#undef RT_REDUCE
    }
    rt_free(work, st);
    return res;
}

template <int LANES>
rt_status shade_lanes(const rt_bvh *bvh, const ShadeDev &S, const float *V, float *rgb, size_t smem, cudaStream_t st) {
    const bool vec = S.K % 4 == 0 && ((uintptr_t)V & 15u) == 0;
    smem += 2 * sizeof(float4) * (size_t)(S.K < kShadeChunk ? S.K : kShadeChunk);
    // a block a multiprocessor always fits, and a small set's call is bound by the
    // host: the occupancy query is 0.3 us of its 8
    const int64_t blocks = (bvh->n * LANES + 127) / 128;
#define RT_SHADE(SH, VEC)                                                                            \
    do {                                                                                             \
        const int64_t cap = blocks <= rt_num_sms()                                                   \
                                ? blocks                                                             \
                                : grid_for((const void *)k_pbr_shade_v<LANES, SH, VEC>, 128, smem);  \
        k_pbr_shade_v<LANES, SH, VEC>                                                                \
            <<<(unsigned)(blocks < cap ? blocks : cap), 128, smem, st>>>(bvh_dev(bvh), S, V, rgb);   \
    } while (0)
    if (S.sh) { if (vec) RT_SHADE(true, true); else RT_SHADE(true, false); }
    else { if (vec) RT_SHADE(false, true); else RT_SHADE(false, false); }
#undef RT_SHADE
    return rt_check_launch();
}

// Threads per Gaussian: the fewest of 1, 4, 16 that give every multiprocessor
// 768 threads (a term is the same work however the terms are dealt out, but
// each thread turns the 27 SH coefficients into its frame for itself), no
// more than a quarter of the terms.
rt_status shade_table(const rt_bvh *bvh, const ShadeDev &S, const float *V, float *rgb, size_t smem, cudaStream_t st) {
    const int64_t want = 768ll * rt_num_sms();
    if (bvh->n >= want || S.K < 16) return shade_lanes<1>(bvh, S, V, rgb, smem, st);
    if (4 * bvh->n >= want || S.K < 64) return shade_lanes<4>(bvh, S, V, rgb, smem, st);
    return shade_lanes<16>(bvh, S, V, rgb, smem, st);
}

}  // namespace

extern "C" rt_status rt_pbr_shade(const rt_bvh *bvh, const rt_rayspec *rays, const float *V,
                                  const rt_pbr_inputs *in, float *rgb, rt_stream_t stream) {
    RaySetDev rs;
    ShadeDev S;
    RT_TRY(shade_dev(bvh, rays, in, &rs, &S));
    if (in->kernel != RT_KERNEL_AUTO && in->kernel != RT_KERNEL_WIDE && in->kernel != RT_KERNEL_RAY_WIDE)
        return RT_ERR_INVALID_ARG;
    if (bvh->n == 0) return RT_OK;
    if (!rgb) return RT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t smem = sizeof(float4) * (size_t)S.env_h * S.env_w;
    if (V) return shade_table(bvh, S, V, rgb, smem, st);
    const int strat = in->kernel == RT_KERNEL_WIDE ? 2 : in->kernel == RT_KERNEL_RAY_WIDE ? 4 : kHemiStrat;
    return launch_reduce<0>(bvh, rs, S, rgb, smem, strat, st);
}

extern "C" rt_status rt_trace_ao(const rt_bvh *bvh, const rt_rayspec *rays, const rt_trace_opts *opts, float *ao,
                                 rt_stream_t stream) {
    const int kernel = opts ? opts->kernel : RT_KERNEL_AUTO;
    if (kernel != RT_KERNEL_AUTO && kernel != RT_KERNEL_WIDE && kernel != RT_KERNEL_RAY_WIDE) return RT_ERR_INVALID_ARG;
    if (!bvh || !rays || rays->ray_ids || (rays->kind != RT_RAYS_DIRS && rays->kind != RT_RAYS_HEMI))
        return RT_ERR_INVALID_ARG;
    RaySetDev rs;
    int64_t count = 0;
    RT_TRY(rt_rayset_dev(bvh, rays, &rs, &count));
    if (bvh->n == 0) return RT_OK;
    if (!ao) return RT_ERR_INVALID_ARG;
    ShadeDev S;
    memset(&S, 0, sizeof(S));
    int strat = rays->kind == RT_RAYS_DIRS && rt_shaft_pays(bvh) ? 3 : kHemiStrat;
    if (kernel == RT_KERNEL_WIDE) strat = rays->kind == RT_RAYS_DIRS ? 3 : 2;
    if (kernel == RT_KERNEL_RAY_WIDE) strat = 4;
    return launch_reduce<1>(bvh, rs, S, ao, 0, strat, (cudaStream_t)stream);
}
