// rt_backward.cu -- adjoint of the visibility trace.
//
// For a ray with final transmittance T = prod_j (1 - alpha_j) and upstream
// gradient g = dL/dT, each accepted Gaussian j receives
//   dL/dalpha_j = -g T / (1 - alpha_j),
//   alpha = o exp(-m^2/2):  dalpha/do = exp(-m^2/2),  dalpha/dm^2 = -alpha/2.
// m^2 is stationary in t at the peak t*, so with the peak point held fixed and
// e = x(t*) - mu, u = S^-1 R^T e, w = S^-1 u:
//   dm^2/dmu = -2 R w,  dm^2/dorigin = +2 R w,  dm^2/ds_k = -2 u_k^2 / s_k,
//   dm^2/dR_ck = 2 e_c w_k, then through R(q/|q|) to the raw quaternion.
// Rays cast from a Gaussian (DIRS / ENV sets) start at mu_src + eps d, so
// their origin gradient is added to the source Gaussian's mean.
// Hits are replayed from the forward's hit log when it is complete for the
// ray, otherwise found again by traversal (same arithmetic as the forward, so
// the same accepted set): a direction set's in shaft packets (ShaftGrad), any
// other ray by ray.  Rays the forward snapped to T = 0 have zero
// gradient.
// Accumulation: float32 atomics into the caller's arrays, or (params
// deterministic = 1) integer atomics on 64-bit fixed point with 2^-32
// resolution, one accumulator per parameter component, added to the caller's
// arrays afterwards: integer addition is associative, so the result does not
// depend on the order in which rays (or shaft groups) finish.
#include <algorithm>

#include "rt_shaft.cuh"

namespace {

struct GradOut {
    float *d_mean, *d_scale, *d_quat, *d_opacity, *d_ray_o;
    const float *mean, *scale, *quat, *opacity;
    long long *fx;  // deterministic mode: [n][kFxPer] fixed-point accumulators
    int *status;
};

// Fixed-point layout per Gaussian: mean 0-2, scale 3-5, quat 6-9, opacity 10.
constexpr int kFxPer = 11;
constexpr float kFxScale = 4294967296.0f;  // 2^32

// v * 2^32 rounded to the nearest integer, added with an integer atomic; a
// value or a sum outside the signed 64-bit range records RT_ERR_RANGE.
__device__ __forceinline__ void fx_add(long long *p, float v, int *status) {
    const float s = v * kFxScale;  // exact: a power of two
    if (!(fabsf(s) < 9.2e18f)) {   // also NaN
        rt_set_error(status, RT_ERR_RANGE);
        return;
    }
    const long long q = __float2ll_rn(s);
    const unsigned long long old = atomicAdd((unsigned long long *)p, (unsigned long long)q);
    const long long o = (long long)old, sum = (long long)(old + (unsigned long long)q);
    if (((o ^ sum) & (q ^ sum)) < 0) rt_set_error(status, RT_ERR_RANGE);
}

template <bool DET>
__device__ __forceinline__ void grad_add(const GradOut &G, float *dst, int64_t i, int slot, float v) {
    if (DET) fx_add(G.fx + i * kFxPer + slot, v, G.status);
    else atomicAdd(dst, v);
}

// Peak point for the gradient: e = x(t*) - mu and alpha with IEEE division
// and exponential.  dm^2/dmu = -2 Sigma^-1 e is first order in e, so t* must
// be accurate here (the forward's accept decision tolerates a fast
// reciprocal because m^2 itself is stationary in t).
__device__ __forceinline__ void peak_accurate(const BvhDev &b, int32_t p, float3 o, float3 d, float &alpha,
                                              float3 &e) {
    const float4x2 r0 = ldg_pair(b.gauss + 4 * (int64_t)p), r1 = ldg_pair(b.gauss + 4 * (int64_t)p + 2);
    const float4 g0 = r0.a, g1 = r0.b, g2 = r1.a, g3 = r1.b;
    float hx, lx, hy, ly, hz, lz;
    two_diff(o.x, g0.x, hx, lx);
    two_diff(o.y, g0.y, hy, ly);
    two_diff(o.z, g0.z, hz, lz);
    const float3 w0 = make_float3(g1.x, g1.y, g1.z);
    const float3 w1 = make_float3(g2.x, g2.y, g2.z);
    const float3 w2 = make_float3(g3.x, g3.y, g3.z);
    const float3 dh = make_float3(hx, hy, hz);
    const float3 ud = make_float3(dot3(w0, d), dot3(w1, d), dot3(w2, d));
    const float3 uo = make_float3(dot3(w0, dh), dot3(w1, dh), dot3(w2, dh));
    const float t = -dot3(uo, ud) / dot3(ud, ud);
    e = make_float3(fmaf(t, d.x, hx) + lx, fmaf(t, d.y, hy) + ly, fmaf(t, d.z, hz) + lz);
    const float3 u = make_float3(dot3(w0, e), dot3(w1, e), dot3(w2, e));
    alpha = g0.w * expf(-0.5f * dot3(u, u));
}

// Gradient contribution of one accepted hit (Gaussian with original index i).
template <bool DET>
__device__ __forceinline__ void hit_grad(const GradOut &G, int32_t i, float gT, float T, float alpha,
                                         float3 e, float3 &d_origin) {
    const float qw0 = G.quat[4 * i], qx0 = G.quat[4 * i + 1], qy0 = G.quat[4 * i + 2], qz0 = G.quat[4 * i + 3];
    const float qn = sqrtf(qw0 * qw0 + qx0 * qx0 + qy0 * qy0 + qz0 * qz0);
    const float w = qw0 / qn, x = qx0 / qn, y = qy0 / qn, z = qz0 / qn;
    float R[3][3];
    R[0][0] = 1.f - 2.f * (y * y + z * z); R[0][1] = 2.f * (x * y - w * z); R[0][2] = 2.f * (x * z + w * y);
    R[1][0] = 2.f * (x * y + w * z); R[1][1] = 1.f - 2.f * (x * x + z * z); R[1][2] = 2.f * (y * z - w * x);
    R[2][0] = 2.f * (x * z - w * y); R[2][1] = 2.f * (y * z + w * x); R[2][2] = 1.f - 2.f * (x * x + y * y);
    const float s[3] = {G.scale[3 * i], G.scale[3 * i + 1], G.scale[3 * i + 2]};
    const float ec[3] = {e.x, e.y, e.z};
    float u[3], wv[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        u[k] = (R[0][k] * ec[0] + R[1][k] * ec[1] + R[2][k] * ec[2]) / s[k];
        wv[k] = u[k] / s[k];
    }
    float sie[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) sie[c] = R[c][0] * wv[0] + R[c][1] * wv[1] + R[c][2] * wv[2];
    const float gA = gT * (-T / (1.0f - alpha));  // dL/dalpha
    const float ex = alpha / G.opacity[i];        // exp(-m^2/2)
    const float gM = gA * (-0.5f * alpha);        // dL/dm^2
    grad_add<DET>(G, G.d_opacity + i, i, 10, gA * ex);
#pragma unroll
    for (int c = 0; c < 3; ++c) grad_add<DET>(G, G.d_mean + 3 * i + c, i, c, -2.0f * gM * sie[c]);
#pragma unroll
    for (int k = 0; k < 3; ++k) grad_add<DET>(G, G.d_scale + 3 * i + k, i, 3 + k, -2.0f * gM * u[k] * u[k] / s[k]);
    float Gm[9];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < 3; ++k) Gm[3 * c + k] = 2.0f * gM * ec[c] * wv[k];
    const float gw = 2.f * (-z * Gm[1] + y * Gm[2] + z * Gm[3] - x * Gm[5] - y * Gm[6] + x * Gm[7]);
    const float gx = 2.f * (y * Gm[1] + z * Gm[2] + y * Gm[3] - 2.f * x * Gm[4] - w * Gm[5] + z * Gm[6] + w * Gm[7] - 2.f * x * Gm[8]);
    const float gy = 2.f * (-2.f * y * Gm[0] + x * Gm[1] + w * Gm[2] + x * Gm[3] + z * Gm[5] - w * Gm[6] + z * Gm[7] - 2.f * y * Gm[8]);
    const float gz = 2.f * (-2.f * z * Gm[0] - w * Gm[1] + x * Gm[2] + w * Gm[3] - 2.f * z * Gm[4] + y * Gm[5] + x * Gm[6] + y * Gm[7]);
    const float dot = w * gw + x * gx + y * gy + z * gz;
    grad_add<DET>(G, G.d_quat + 4 * i + 0, i, 6, (gw - w * dot) / qn);
    grad_add<DET>(G, G.d_quat + 4 * i + 1, i, 7, (gx - x * dot) / qn);
    grad_add<DET>(G, G.d_quat + 4 * i + 2, i, 8, (gy - y * dot) / qn);
    grad_add<DET>(G, G.d_quat + 4 * i + 3, i, 9, (gz - z * dot) / qn);
    d_origin.x += 2.0f * gM * sie[0];
    d_origin.y += 2.0f * gM * sie[1];
    d_origin.z += 2.0f * gM * sie[2];
}

template <bool DET>
__global__ void __launch_bounds__(128) k_backward(BvhDev b, RaySetDev rs, int64_t R, const float *T,
                                                  const float *dL_dT, const int32_t *hit_ids,
                                                  const int32_t *hit_count, int32_t cap, GradOut G,
                                                  int *status) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < R;
         r += (int64_t)gridDim.x * blockDim.x) {
        float3 o, d;
        int32_t src = -1;      // sorted position of the excluded Gaussian
        int32_t src_orig = -1; // its original index (implicit sets)
        if (rs.kind == RT_RAYS_EXPLICIT) {
            o = make_float3(rs.ray_o[3 * r], rs.ray_o[3 * r + 1], rs.ray_o[3 * r + 2]);
            d = make_float3(rs.ray_d[3 * r], rs.ray_d[3 * r + 1], rs.ray_d[3 * r + 2]);
            if (rs.ray_src) {
                const int32_t s = rs.ray_src[r];
                src = (s >= 0 && s < b.n) ? b.rank[s] : -1;
            }
        } else {
            const int64_t rid = rs.ray_ids ? rs.ray_ids[r] : r;
            if (rid < 0 || rid >= rs.n_rays) {
                rt_set_error(status, RT_ERR_INVALID_ARG);
                continue;
            }
            const int64_t g = rid / rs.K;
            const int32_t k = (int32_t)(rid - g * rs.K);
            src = b.rank[g];
            src_orig = (int32_t)g;
            implicit_ray(rs, rid, k, g, __ldg(b.gauss + 4 * (int64_t)src), o, d);
        }
        float3 d_origin = make_float3(0.f, 0.f, 0.f);
        const float Tr = T[r];
        const float gT = dL_dT[r];
        const bool live = gT != 0.0f && !(b.t_min > 0.0f && Tr == 0.0f);
        if (live) {
            const int32_t cnt = hit_count ? hit_count[r] : -1;
            if (hit_ids && cnt >= 0 && cnt <= cap) {
                for (int32_t h = 0; h < cnt; ++h) {  // the forward accepted these: no re-check
                    const int32_t i = hit_ids[r * (int64_t)cap + h];
                    const int32_t p = b.rank[i];
                    float alpha;
                    float3 e;
                    peak_accurate(b, p, o, d, alpha, e);
                    hit_grad<DET>(G, i, gT, Tr, alpha, e, d_origin);
                }
            } else if (b.n == 1) {
                float alpha;
                float3 e;
                if (src != 0 && gauss_eval(b, 0, o, d, alpha, e)) {
                    peak_accurate(b, 0, o, d, alpha, e);
                    hit_grad<DET>(G, __float_as_int(__ldg(b.gauss + 1).w), gT, Tr, alpha, e, d_origin);
                }
            } else if (b.n > 1) {
                const float3 inv = safe_inv(d);
                const float3 oi = make_float3(o.x * inv.x, o.y * inv.y, o.z * inv.z);
                uint32_t stack[RT_STACK];
                int sp = 0;
                uint32_t node = 0;
                for (;;) {
                    const float4x2 q0 = ldg_pair(b.nodes + 4 * (int64_t)node), q1 = ldg_pair(b.nodes + 4 * (int64_t)node + 2);
                    const float4 n0 = q0.a, n1 = q0.b, n2 = q1.a, n3 = q1.b;
                    bool hl = slab(n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, oi, inv);
                    bool hr = slab(n1.z, n1.w, n2.x, n2.y, n2.z, n2.w, oi, inv);
                    const uint32_t ch[2] = {__float_as_uint(n3.x), __float_as_uint(n3.y)};
                    bool hit2[2] = {hl, hr};
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        if (hit2[c] && (ch[c] & RT_LEAF_BIT)) {
                            hit2[c] = false;
                            const int32_t p = (int32_t)(ch[c] & ~RT_LEAF_BIT);
                            float alpha;
                            float3 e;
                            if (p != src && gauss_eval(b, p, o, d, alpha, e)) {  // the forward's decision
                                peak_accurate(b, p, o, d, alpha, e);
                                hit_grad<DET>(G, __float_as_int(__ldg(b.gauss + 4 * p + 1).w), gT, Tr, alpha,
                                              e, d_origin);
                            }
                        }
                    }
                    if (hit2[0] && hit2[1]) {
                        if (sp >= RT_STACK) {
                            rt_set_error(status, RT_ERR_STACK_OVERFLOW);
                            break;
                        }
                        stack[sp++] = ch[1];
                        node = ch[0];
                    } else if (hit2[0]) {
                        node = ch[0];
                    } else if (hit2[1]) {
                        node = ch[1];
                    } else {
                        if (sp == 0) break;
                        node = stack[--sp];
                    }
                }
            }
        }
        if (G.d_ray_o) {
            G.d_ray_o[3 * r] = d_origin.x;
            G.d_ray_o[3 * r + 1] = d_origin.y;
            G.d_ray_o[3 * r + 2] = d_origin.z;
        }
        if (src_orig >= 0 && live) {
            grad_add<DET>(G, G.d_mean + 3 * src_orig, src_orig, 0, d_origin.x);
            grad_add<DET>(G, G.d_mean + 3 * src_orig + 1, src_orig, 1, d_origin.y);
            grad_add<DET>(G, G.d_mean + 3 * src_orig + 2, src_orig, 2, d_origin.z);
        }
    }
}

// A direction set whose groups pay (rt_shaft_pays) and no hit log: one warp
// per group and direction finds the hits of the group's rays as the forward's
// shaft packets do and sums what each Gaussian receives over those rays before
// anything leaves the SM.  With u = S^-1 R^T e and g = dL/dm^2 of each hit,
//   S0 = sum g, v = sum g u, M = sum g u u^T
// hold all of a Gaussian's gradient:
//   do = -2 S0 / o,  dmu = -2 R S^-1 v,  ds_k = -2 M_kk / s_k,
//   dR = 2 R L, L_jk = M_jk s_j / s_k: the quaternion's gradient is
//   2 q x (0, tau) / |q| with tau the antisymmetric part of L twice,
//   tau_x = 2 M_12 (s_2 / s_1 - s_1 / s_2) and so on,
// and a ray's origin receives 2 g W^T u of each hit, W = S^-1 R^T (the record).
// The sums run in float32 in the rays' order, so they are the same in every
// run; they go out as float32 or fixed-point atomics as everywhere.  Error
// against float64 as before (uniform 4k scene, relative norm 6.6e-6 both).
//
// What it replaces: a replay of the forward's hit log with 11 atomics per hit
// (bound by those: 17.5M hits of 50k Gaussians x 32, 3.1 ms with fixed-point
// sums, 1.5 ms float32) and the log itself, which cost the forward 1.2 ms.
// This takes 1.77 / 1.54 ms with 3.4 hits per Gaussian summed before the
// atomics.  Bound: instruction issue (0.52 of the slots, 16 warps an SM), then
// waits for instructions (the code is long) and memory.  Measured on the way
// (50k, fixed point): Gaussians hit closed up before their atomics, and those
// all under way before the first result is looked at 3.05 -> 2.44 ms; 4
// resident blocks of 128 registers instead of 5 of 96 2.24 -> 1.77; both
// Gaussians of a lane summed in one loop 2.01 -> 1.77; lists of 256 pairs
// instead of 160 1.77 -> 2.03.
static_assert(4 * kShaftPairs<true> >= 10 * kShaftCands && kShaftPairs<true> < 256, "sums and pair numbers");
template <bool DET>
struct ShaftGrad {
    GradOut G;
    const float *T, *dL_dT;
    int32_t K, k;
    bool snap;
    int live;         // slots: rays with a gradient
    float3 d_org[2];  // of slots lane and lane + 32

    __device__ __forceinline__ int64_t ray(const BvhDev &b, int64_t p) const {
        return (int64_t)__float_as_int(__ldg(b.gauss + 4 * p + 1).w) * K + k;
    }
    // dL/dT T of ray i of the group; false if it has no gradient
    __device__ __forceinline__ float load(const BvhDev &b, int64_t first, int i, bool &in) {
        d_org[0] = d_org[1] = make_float3(0.f, 0.f, 0.f);
        if (!in) return 0.0f;
        const int64_t r = ray(b, first + i);
        const float t = T[r], g = dL_dT[r];
        in = g != 0.0f && !(snap && t == 0.0f);
        if (!in && G.d_ray_o) {
            G.d_ray_o[3 * r] = 0.0f;
            G.d_ray_o[3 * r + 1] = 0.0f;
            G.d_ray_o[3 * r + 2] = 0.0f;
        }
        return g * t;
    }
    // v[0..N) to accumulator slots slot, slot + 1, ... of Gaussian i.  The
    // fixed-point sums are read back by the atomics (range check): all are
    // under way before the first is looked at.
    template <int N>
    __device__ __forceinline__ void add_fx(int64_t i, int slot, const float (&v)[N]) const {
        long long q[N], old[N];
        bool bad = false;
#pragma unroll
        for (int c = 0; c < N; ++c) {
            const float s = v[c] * kFxScale;
            const bool ok = fabsf(s) < 9.2e18f;
            bad |= !ok;
            q[c] = __float2ll_rn(ok ? s : 0.0f);
            old[c] = (long long)atomicAdd((unsigned long long *)(G.fx + i * kFxPer + slot + c), (unsigned long long)q[c]);
        }
#pragma unroll
        for (int c = 0; c < N; ++c) {
            const long long sum = (long long)((unsigned long long)old[c] + (unsigned long long)q[c]);
            bad |= ((old[c] ^ sum) & (q[c] ^ sum)) < 0;
        }
        if (bad) rt_set_error(G.status, RT_ERR_RANGE);
    }
    // A Gaussian's sums to the caller's arrays.
    __device__ __forceinline__ void flush(int64_t i, const float (&S)[10]) const {
        const float q0 = G.quat[4 * i], q1 = G.quat[4 * i + 1], q2 = G.quat[4 * i + 2], q3 = G.quat[4 * i + 3];
        const float iq = 1.0f / sqrtf(q0 * q0 + q1 * q1 + q2 * q2 + q3 * q3);
        const float w = q0 * iq, x = q1 * iq, y = q2 * iq, z = q3 * iq;
        const float s0 = G.scale[3 * i], s1 = G.scale[3 * i + 1], s2 = G.scale[3 * i + 2];
        const float i0 = 1.0f / s0, i1 = 1.0f / s1, i2 = 1.0f / s2;
        const float v0 = -2.f * S[1] * i0, v1 = -2.f * S[2] * i1, v2 = -2.f * S[3] * i2;
        // M_jk (s_j / s_k - s_k / s_j) without a difference of quotients
        const float tx = 2.f * S[8] * ((s2 - s1) * i1 * ((s2 + s1) * i2)),
                    ty = 2.f * S[6] * ((s0 - s2) * i0 * ((s0 + s2) * i2)),
                    tz = 2.f * S[5] * ((s1 - s0) * i0 * ((s1 + s0) * i1));
        const float f = 2.f * iq;
        const float v[kFxPer] = {
            (1.f - 2.f * (y * y + z * z)) * v0 + 2.f * (x * y - w * z) * v1 + 2.f * (x * z + w * y) * v2,
            2.f * (x * y + w * z) * v0 + (1.f - 2.f * (x * x + z * z)) * v1 + 2.f * (y * z - w * x) * v2,
            2.f * (x * z - w * y) * v0 + 2.f * (y * z + w * x) * v1 + (1.f - 2.f * (x * x + y * y)) * v2,
            -2.f * S[4] * i0, -2.f * S[7] * i1, -2.f * S[9] * i2,
            -f * (x * tx + y * ty + z * tz), f * (w * tx + y * tz - z * ty), f * (w * ty + z * tx - x * tz),
            f * (w * tz + x * ty - y * tx),
            -2.f * S[0] / G.opacity[i]};
        if (DET) {
            add_fx(i, 0, v);
        } else {
#pragma unroll
            for (int c = 0; c < 3; ++c) atomicAdd(G.d_mean + 3 * i + c, v[c]);
#pragma unroll
            for (int c = 0; c < 3; ++c) atomicAdd(G.d_scale + 3 * i + c, v[3 + c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) atomicAdd(G.d_quat + 4 * i + c, v[6 + c]);
            atomicAdd(G.d_opacity + i, v[10]);
        }
    }
    // The hits of a batch: m Gaussians (records in sm.stage, sorted positions
    // leaf[0..m)), votes by slot in sm.mask and, for the Gaussians lane and
    // lane + 32, by slot bit in ca and cb.
    __device__ __forceinline__ void batch(const BvhDev &b, float3 d, int64_t first, int n_slots, int m,
                                          const uint32_t *leaf, uint2 ca, uint2 cb, ShaftSmem<true> &sm) {
        const unsigned FULL = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        const unsigned lt = (1u << lane) - 1u;
        auto rec = [&](int i, int r) { return sm.stage[4 * i + (r ^ ((i >> 1) & 3))]; };
        float A[2][10];  // sums of Gaussians lane, lane + 32
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 10; ++c) A[r][c] = 0.0f;
#pragma unroll 1
        for (int s0 = 0; s0 < n_slots; s0 += 32) {
            uint2 mk = make_uint2(0u, 0u);
            if (s0 + lane < n_slots) {
                mk = sm.mask[s0 + lane];
                mk.x &= m >= 32 ? FULL : (1u << m) - 1u;  // a NaN test passes: not past the batch
                mk.y &= m >= 64 ? FULL : m > 32 ? (1u << (m - 32)) - 1u : 0u;
            }
            const int cnt = __popc(mk.x) + __popc(mk.y);
            int end = cnt;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int v = __shfl_up_sync(FULL, end, off);
                if (lane >= off) end += v;
            }
            const int total = __shfl_sync(FULL, end, 31);
            // as many slots at a time as the list holds (64 pairs each at most)
            for (int base = 0, t0 = 0; base < total;) {
                const unsigned fit = __ballot_sync(FULL, end - base <= kShaftPairs<true>);
                const int t1 = __popc(fit), part = __shfl_sync(FULL, end, t1 - 1) - base;
                const bool mine = lane >= t0 && lane < t1;
                if (mine) {
                    int at = end - cnt - base;
                    sm.from[s0 + lane] = (uint8_t)at;
                    for (uint32_t v = mk.x; v; v &= v - 1u)
                        sm.pair[at++].x = __uint_as_float((uint32_t)(s0 + lane) << 6 | (uint32_t)(__ffs(v) - 1));
                    for (uint32_t v = mk.y; v; v &= v - 1u)
                        sm.pair[at++].x = __uint_as_float((uint32_t)(s0 + lane) << 6 | (uint32_t)(__ffs(v) + 31));
                }
                __syncwarp();
#pragma unroll 1
                for (int i = lane; i < part; i += 64) {
                    const bool two = i + 32 < part;
                    const uint32_t pa = __float_as_uint(sm.pair[i].x),
                                   pb = two ? __float_as_uint(sm.pair[i + 32].x) : pa;
                    const int qa = pa & 63u, qb = pb & 63u;
                    const float4 oa = sm.ro[pa >> 6], ob = sm.ro[pb >> 6];
                    const float4 ra[4] = {rec(qa, 0), rec(qa, 1), rec(qa, 2), rec(qa, 3)};
                    const float4 rb[4] = {rec(qb, 0), rec(qb, 1), rec(qb, 2), rec(qb, 3)};
                    PairEval e(b, ra, rb, oa, ob, d);
                    // the ray's own Gaussian
                    if (leaf[qa] == (uint32_t)first + sm.live[pa >> 6]) e.acc[0] = false;
                    if (leaf[qb] == (uint32_t)first + sm.live[pb >> 6]) e.acc[1] = false;
                    // u and alpha at the accurate peak (see peak_accurate)
                    const f2x3 u = e.whiten(e.peak(make_float2(-e.num.x / e.den.x, -e.num.y / e.den.y)));
                    const float2 m2 = e.dot(u, u);
                    const float aa = ra[0].w * expf(-0.5f * m2.x), ab = rb[0].w * expf(-0.5f * m2.y);
                    // dL/dm^2 = dL/dalpha (-alpha / 2), dL/dalpha = -dL/dT T / (1 - alpha)
                    const float ga = 0.5f * aa * (oa.w / (1.0f - aa)), gb = 0.5f * ab * (ob.w / (1.0f - ab));
                    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
                    sm.pair[i] = e.acc[0] ? make_float4(ga, u.x.x, u.y.x, u.z.x) : zero;
                    if (two) sm.pair[i + 32] = e.acc[1] ? make_float4(gb, u.x.y, u.y.y, u.z.y) : zero;
                }
                __syncwarp();
                if (mine) {  // the rays' origins
                    float3 a = make_float3(0.f, 0.f, 0.f);
                    int at = end - cnt - base;
                    uint64_t v = (uint64_t)mk.y << 32 | mk.x;
#pragma unroll 2
                    while (v) {
                        const float4 p = sm.pair[at++];
                        const int c = __ffsll((long long)v) - 1;
                        v &= v - 1ull;
                        const float4 w0 = rec(c, 1), w1 = rec(c, 2), w2 = rec(c, 3);
                        const float g = 2.0f * p.x;
                        a.x = fmaf(g, fmaf(w0.x, p.y, fmaf(w1.x, p.z, w2.x * p.w)), a.x);
                        a.y = fmaf(g, fmaf(w0.y, p.y, fmaf(w1.y, p.z, w2.y * p.w)), a.y);
                        a.z = fmaf(g, fmaf(w0.z, p.y, fmaf(w1.z, p.z, w2.z * p.w)), a.z);
                    }
                    if (s0 == 0) {
                        d_org[0].x += a.x;
                        d_org[0].y += a.y;
                        d_org[0].z += a.z;
                    } else {
                        d_org[1].x += a.x;
                        d_org[1].y += a.y;
                        d_org[1].z += a.z;
                    }
                }
                // the Gaussians, each over its slots of this part
                const uint32_t range = (t1 >= 32 ? FULL : (1u << t1) - 1u) & ~((1u << t0) - 1u);
                uint32_t v[2] = {(s0 == 0 ? ca.x : ca.y) & range, (s0 == 0 ? cb.x : cb.y) & range};
                while (v[0] | v[1]) {
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const bool on = v[r] != 0u;
                        const int t = s0 + (on ? __ffs(v[r]) - 1 : t0);
                        v[r] &= v[r] - 1u;
                        const uint2 mt = sm.mask[t];
                        const int at = sm.from[t] + (r == 0 ? __popc(mt.x & lt) : __popc(mt.x) + __popc(mt.y & lt));
                        float4 p = sm.pair[on ? at : 0];
                        float(&S)[10] = A[r];
                        p.x = on ? p.x : 0.0f;
                        const float gx = p.x * p.y, gy = p.x * p.z, gz = p.x * p.w;
                        S[0] += p.x;
                        S[1] += gx;
                        S[2] += gy;
                        S[3] += gz;
                        S[4] = fmaf(gx, p.y, S[4]);
                        S[5] = fmaf(gx, p.z, S[5]);
                        S[6] = fmaf(gx, p.w, S[6]);
                        S[7] = fmaf(gy, p.z, S[7]);
                        S[8] = fmaf(gy, p.w, S[8]);
                        S[9] = fmaf(gz, p.w, S[9]);
                    }
                }
                __syncwarp();
                base += part;
                t0 = t1;
            }
        }
        // the Gaussians hit, closed up: sums c at [c][slot], over the pair list
        float *sums = &sm.pair[0].x;
        unsigned hit[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            bool any = false;
#pragma unroll
            for (int c = 0; c < 10; ++c) any |= A[r][c] != 0.0f;  // only Gaussians of the batch
            hit[r] = __ballot_sync(FULL, any);
            if (any) {
                const int at = __popc(hit[r] & lt) + (r == 0 ? 0 : __popc(hit[0]));
                sm.from[at] = (uint8_t)(lane + 32 * r);
#pragma unroll
                for (int c = 0; c < 10; ++c) sums[c * kShaftCands + at] = A[r][c];
            }
        }
        __syncwarp();
        const int n_hit = __popc(hit[0]) + __popc(hit[1]);
#pragma unroll 1
        for (int i = lane; i < n_hit; i += 32) {
            float S[10];
#pragma unroll
            for (int c = 0; c < 10; ++c) S[c] = sums[c * kShaftCands + i];
            flush(__float_as_int(rec(sm.from[i], 1).w), S);
        }
        __syncwarp();
    }
    __device__ __forceinline__ void finish(const BvhDev &b, int64_t first, const ShaftSmem<true> &sm) const {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (lane + 32 * r >= live) continue;
            const int64_t i = ray(b, first + sm.live[lane + 32 * r]), g = i / K;
            if (G.d_ray_o) {
                G.d_ray_o[3 * i] = d_org[r].x;
                G.d_ray_o[3 * i + 1] = d_org[r].y;
                G.d_ray_o[3 * i + 2] = d_org[r].z;
            }
            const float v[3] = {d_org[r].x, d_org[r].y, d_org[r].z};
            if (DET) {
                add_fx(g, 0, v);
            } else {
#pragma unroll
                for (int c = 0; c < 3; ++c) atomicAdd(G.d_mean + 3 * g + c, v[c]);
            }
        }
    }
};

template <bool DET>
__global__ void __launch_bounds__(128, 4) k_shaft_backward(BvhDev b, RaySetDev rs, int64_t n_items,
                                                                            ShaftGrad<DET> init, int *status,
                                                                            unsigned long long *work) {
    __shared__ ShaftSmem<true> sm_all[4];
    ShaftSmem<true> &sm = sm_all[threadIdx.x >> 5];
    for (;;) {
        unsigned long long item = 0;
        if ((threadIdx.x & 31) == 0) item = atomicAdd(work, 1ull);
        item = __shfl_sync(0xffffffffu, item, 0);
        if ((int64_t)item >= n_items) break;
        const int64_t gi = (int64_t)item / rs.K;
        const int32_t k = (int32_t)((int64_t)item - gi * rs.K);
        const int2 gr = __ldg(b.groups + gi);
        ShaftGrad<DET> g = init;
        g.k = k;
        shaft_group<true>(b, rs.eps, make_float3(__ldg(rs.dirs + 3 * k), __ldg(rs.dirs + 3 * k + 1), __ldg(rs.dirs + 3 * k + 2)),
                          gr.x, gr.y, status, sm, &g);
        __syncwarp();
        g.finish(b, gr.x, sm);
        __syncwarp();
    }
}

// Deterministic mode: adds the fixed-point sums (times 2^-32) to the caller's
// arrays.
__global__ void k_fx_finalize(const long long *__restrict__ fx, int64_t n, float *d_mean, float *d_scale,
                              float *d_quat, float *d_opacity) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n * kFxPer;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = j / kFxPer;
        const int c = (int)(j - i * kFxPer);
        const float v = (float)((double)fx[j] * (1.0 / 4294967296.0));
        if (c < 3) d_mean[3 * i + c] += v;
        else if (c < 6) d_scale[3 * i + c - 3] += v;
        else if (c < 10) d_quat[4 * i + c - 6] += v;
        else d_opacity[i] += v;
    }
}

template <bool DET>
void launch_shafts(const BvhDev &b, const RaySetDev &rs, int64_t n_groups, const GradOut &G, const float *T,
                   const float *dL_dT, unsigned long long *work, cudaStream_t st) {
    ShaftGrad<DET> g;
    g.G = G;
    g.T = T;
    g.dL_dT = dL_dT;
    g.K = rs.K;
    g.k = 0;
    g.snap = b.t_min > 0.0f;
    g.live = 0;
    g.d_org[0] = g.d_org[1] = make_float3(0.f, 0.f, 0.f);
    const int64_t items = n_groups * rs.K;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_shaft_backward<DET>, 128, 0) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    const int64_t grid = std::min<int64_t>((items + 3) / 4, (int64_t)per_sm * rt_num_sms());
    k_shaft_backward<DET><<<(int)grid, 128, 0, st>>>(b, rs, items, g, G.status, work);
}

// A full direction set whose groups pay takes the shaft packets.
bool rt_backward_shafts(const rt_bvh *bvh, const rt_rayspec *rays) {
    return rays->kind == RT_RAYS_DIRS && !rays->ray_ids && rt_shaft_pays(bvh);
}

}  // namespace

// With a log the forward walks ray by ray.  Forward + adjoint of 32 directions,
// us, shafts against log: 8 rays a group or more (uniform 4k, 10 rays: 359 /
// 450; uniform 30k: 2,692 / 9,940; object 50k: 2,404 / 3,587); below (object
// 20k, 7 rays) 1,078 / 906, or 1,168 / 1,424 with fixed-point sums, of which
// the log's replay has one per hit.
extern "C" int32_t rt_backward_wants_log(const rt_bvh *bvh, const rt_rayspec *rays) {
    if (!bvh || !rays) return 0;
    return !(rt_backward_shafts(bvh, rays) && (bvh->params.deterministic || bvh->n >= 8 * bvh->n_groups));
}

extern "C" rt_status rt_trace_visibility_backward(const rt_bvh *bvh, const rt_rayspec *rays,
                                                  const float *mean, const float *scale,
                                                  const float *quat, const float *opacity,
                                                  const float *T, const float *dL_dT,
                                                  const int32_t *hit_ids, const int32_t *hit_count,
                                                  int32_t hit_cap, float *d_mean, float *d_scale,
                                                  float *d_quat, float *d_opacity, float *d_ray_o,
                                                  rt_stream_t stream) {
    if (!bvh || !rays) return RT_ERR_INVALID_ARG;
    RaySetDev rs;
    int64_t R = 0;
    RT_TRY(rt_rayset_dev(bvh, rays, &rs, &R));
    if (R == 0 || bvh->n == 0) return RT_OK;
    if (!mean || !scale || !quat || !opacity || !T || !dL_dT || !d_mean || !d_scale || !d_quat || !d_opacity)
        return RT_ERR_INVALID_ARG;
    if (hit_ids && (!hit_count || hit_cap <= 0)) return RT_ERR_INVALID_ARG;
    GradOut G;
    G.d_mean = d_mean;
    G.d_scale = d_scale;
    G.d_quat = d_quat;
    G.d_opacity = d_opacity;
    G.d_ray_o = d_ray_o;
    G.mean = mean;
    G.scale = scale;
    G.quat = quat;
    G.opacity = opacity;
    G.fx = nullptr;
    G.status = rt_status_ptr();
    int64_t grid = (R + 127) / 128;
    const int64_t cap_grid = (int64_t)rt_num_sms() * 16;
    if (grid > cap_grid) grid = cap_grid;
    cudaStream_t st = (cudaStream_t)stream;
    const bool det = bvh->params.deterministic != 0;
    bool shafts = !hit_ids && rt_backward_shafts(bvh, rays);
    // scratch: the fixed-point sums and the shafts' work counter
    const size_t fx_bytes = det ? ((size_t)bvh->n * kFxPer * sizeof(long long)) : 0;
    char *blk = nullptr;
    if (det || shafts) {
        const rt_status a = rt_alloc((void **)&blk, fx_bytes + (shafts ? 8 : 0), stream);
        if (a != RT_OK && det) return a;
        if (a != RT_OK) shafts = false;  // the per-ray kernel needs none
    }
    rt_status s = RT_OK;
    if (blk && cudaMemsetAsync(blk, 0, fx_bytes + (shafts ? 8 : 0), st) != cudaSuccess) {
        cudaGetLastError();
        s = RT_ERR_CUDA;
    }
    if (s == RT_OK) {
        if (det) G.fx = (long long *)blk;
        const BvhDev b = bvh_dev(bvh);
        unsigned long long *work = (unsigned long long *)(blk + fx_bytes);
        if (shafts) {
            if (det) launch_shafts<true>(b, rs, bvh->n_groups, G, T, dL_dT, work, st);
            else launch_shafts<false>(b, rs, bvh->n_groups, G, T, dL_dT, work, st);
        } else if (det) {
            k_backward<true><<<(int)grid, 128, 0, st>>>(b, rs, R, T, dL_dT, hit_ids, hit_count, hit_cap, G, G.status);
        } else {
            k_backward<false><<<(int)grid, 128, 0, st>>>(b, rs, R, T, dL_dT, hit_ids, hit_count, hit_cap, G, G.status);
        }
        if (det) {
            int64_t fgrid = (bvh->n * kFxPer + 255) / 256;
            if (fgrid > (int64_t)rt_num_sms() * 8) fgrid = (int64_t)rt_num_sms() * 8;
            k_fx_finalize<<<(int)fgrid, 256, 0, st>>>(G.fx, bvh->n, d_mean, d_scale, d_quat, d_opacity);
        }
        s = rt_check_launch();
    }
    if (blk) rt_free(blk, stream);
    return s;
}
