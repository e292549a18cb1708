// rt_shaft.cuh -- shaft packets: visibility of the parallel rays that a group
// of neighbouring Gaussians casts along one direction of a direction set.
//
// A group (at most 64 consecutive sorted positions, rt_bvh's groups) and a
// direction sweep a narrow shaft.  One warp walks the tree for the whole
// shaft; its lanes are split over what each step has most of:
//   1. nodes: up to 16 nodes at a time come off a shared stack, two lanes
//      per 64-byte node test its boxes against the shaft: the ray from the
//      centre of the origins' box against boxes grown by that box's half
//      extents (the Minkowski sum, exact for parallel rays).  Leaves met go to
//      a list.
//   2. Gaussians: 64 leaves at a time, two per lane (packed FMAs).  A lane
//      reduces its Gaussians to what is left of them along d: a whitened 2D
//      offset v = (r11 x + r12 y + c1, r22 y + c2) of the ray through (x, y)
//      of the plane across d, |v|^2 = m^2 log2(e)/2, and the plane t* = 0.
//      The live rays pass by, one vote each: the Gaussians it may accept.
//   3. (ray, Gaussian) pairs: the votes are written out as a list and
//      evaluated 64 at a time (two per lane, packed FMAs) with the arithmetic
//      of gauss_eval, the records read from shared memory; each ray then
//      multiplies its factors into its T.
// The float32 test of step 2 only rejects: its limits are widened by a bound
// on its own rounding and on gauss_eval's (an unordered compare passes), so
// the accepted set is that of the other strategies; only the order of the
// factors differs.  Finished rays leave the group, and each time a quarter of
// them has, the shaft is drawn in around the rest (2M scene: 14 % faster).
//
// What it replaces: the packet walk with one box test per ray and node issued
// 182k warp instructions per 32 rays of the 2M-Gaussian object scene (307 per
// node visit, of which a ray needs half); this takes ~28k, 0.7 of them in
// steps 1 and 3.  Measured, trace only, against that walk (2M x 64
// directions: 751 -> 123 ms, 1.0 G rays/s) and the per-ray walk (300k x 128:
// 96 -> 26.5 ms, 1.45 G rays/s).  Bound: instruction issue (0.7 of the slots;
// the rest fixed-latency dependences), with shared memory at 0.65 of its
// wavefronts; DRAM 0.1 %.  Choices measured on the way (300k / 2M scenes):
//   - records staged by 4 lanes each with 16-byte async copies: with a 16-byte
//     load per lane and row the kernel was bound by L1 tag lookups (91 %);
//   - 64-byte nodes in two 32-byte loads a lane instead of 128-byte ones staged
//     like the records: 4 to 6 % (300k x 32 7.07 -> 6.68 ms, 50k x 32 875 -> 825
//     us); one lane per node, 32 a step: 50k 946 us;
//   - pairs evaluated from a list: with each ray walking its own mask, 9 of
//     32 lanes were busy; writing the list from the voting lanes instead of
//     the rays' masks was 10 % slower;
//   - groups of up to 64 rays instead of tiles of 32 (20 %), cut at the jumps
//     of the Morton curve (an uncut jump makes one warp walk the whole scene:
//     2M 2.2x slower);
//   - 6 resident blocks (80 registers) instead of 5 (96): 6 %.
#pragma once

#include <type_traits>

#include "rt_trace_core.cuh"

constexpr int kShaftRays = 64;      // rays of a group at most
constexpr int kShaftCands = 64;     // Gaussians of a batch
constexpr int kShaftNodes = 16;     // nodes of a step
constexpr int kShaftLeaves = 128;   // leaves met: fewer than a batch left over and a step's
constexpr int kShaftStack = 320;    // nodes; a walk of single nodes adds 3 per level at most (193 for 64 levels)
template <bool GRAD>
constexpr int kShaftPairs = GRAD ? 160 : 256;

// The adjoint (GRAD) keeps a record per pair, (dL/dm^2, u) with u = S^-1 R^T e.
template <bool GRAD>
struct __align__(16) ShaftSmem {
    float4 stage[4 * kShaftCands];            // the batch's records
    float4 ro[kShaftRays];                    // by ray: origin, T (GRAD: by slot: origin, dL/dT T)
    typename std::conditional<GRAD, float4, uint32_t>::type pair[kShaftPairs<GRAD>];  // ray << 6 | Gaussian,
                                              //   then the pair's factor (GRAD: record)
    float2 xy[kShaftRays];                    // by slot of a live ray: its place across d
    float z[kShaftRays];                      //   and along d
    uint2 mask[kShaftRays];                   // by slot: Gaussians of the batch to evaluate
    float4 fr[5];                             // the shaft's frame (see shaft_cand)
    uint32_t stack[kShaftStack];
    uint32_t leaf[kShaftLeaves];
    uint8_t live[kShaftRays];                 // by slot: ray
    uint8_t from[GRAD ? kShaftRays : 1];      // GRAD: by slot: its first pair
};

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ uint32_t float_ord(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord_float(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}
__device__ __forceinline__ float warp_min(float v) {
    return ord_float(__reduce_min_sync(0xffffffffu, float_ord(v)));
}
__device__ __forceinline__ float warp_max(float v) {
    return ord_float(__reduce_max_sync(0xffffffffu, float_ord(v)));
}

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }
struct f2x3 {
    float2 x, y, z;
};
__device__ __forceinline__ f2x3 pack3(float4 a, float4 b) {
    f2x3 r;
    r.x = make_float2(a.x, b.x);
    r.y = make_float2(a.y, b.y);
    r.z = make_float2(a.z, b.z);
    return r;
}
__device__ __forceinline__ float2 dot2(f2x3 a, f2x3 b) {
    return __ffma2_rn(a.x, b.x, __ffma2_rn(a.y, b.y, __fmul2_rn(a.z, b.z)));
}
__device__ __forceinline__ float2 dot2(f2x3 a, float4 b) {
    return __ffma2_rn(a.x, dup(b.x), __ffma2_rn(a.y, dup(b.y), __fmul2_rn(a.z, dup(b.z))));
}

// Children 2 h and 2 h + 1 of a 64-byte node against a shaft (see qnode_near):
// the near planes moved towards the rays by the origins' half extents and the
// far planes away (cn, cf = c inv +- hh |inv|).
__device__ __forceinline__ void shaft_qnode(const float4 *__restrict__ q, int h, float3 inv, float3 cn, float3 cf,
                                            bool &h0, bool &h1, uint32_t &r0, uint32_t &r1) {
    const float4x2 n0 = ldg_pair(q), n1 = ldg_pair(q + 2);
    const float ax = n0.a.w * inv.x, ay = n0.b.x * inv.y, az = n0.b.y * inv.z;
    const float nx = fmaf(n0.a.x, inv.x, -cn.x), ny = fmaf(n0.a.y, inv.y, -cn.y), nz = fmaf(n0.a.z, inv.z, -cn.z);
    const float fx = fmaf(n0.a.x, inv.x, -cf.x), fy = fmaf(n0.a.y, inv.y, -cf.y), fz = fmaf(n0.a.z, inv.z, -cf.z);
    const bool sx = inv.x < 0.0f, sy = inv.y < 0.0f, sz = inv.z < 0.0f;
    const uint32_t lx = __float_as_uint(n0.b.z), hx = __float_as_uint(n0.b.w), ly = __float_as_uint(n1.a.x),
                   hy = __float_as_uint(n1.a.y), lz = __float_as_uint(n1.a.z), hz = __float_as_uint(n1.a.w);
    r0 = __float_as_uint(h ? n1.b.z : n1.b.x);
    r1 = __float_as_uint(h ? n1.b.w : n1.b.y);
    const uint32_t s0 = h ? 0x7624u : 0x7604u, s1 = s0 + 0x10u;
    auto dist = [&](uint32_t w, float a, float c) {
        const float2 k = make_float2(__uint_as_float(__byte_perm(w, 0x3f800000u, s0)),
                                     __uint_as_float(__byte_perm(w, 0x3f800000u, s1)));
        return __ffma2_rn(k, make_float2(a, a), make_float2(c, c));
    };
    const float2 x0 = dist(sx ? hx : lx, ax, nx), x1 = dist(sx ? lx : hx, ax, fx), y0 = dist(sy ? hy : ly, ay, ny),
                 y1 = dist(sy ? ly : hy, ay, fy), z0 = dist(sz ? hz : lz, az, nz), z1 = dist(sz ? lz : hz, az, fz);
    const float na = fmaxf(fmaxf(x0.x, y0.x), fmaxf(z0.x, 0.0f)), fa = fminf(fminf(x1.x, y1.x), z1.x);
    const float nb = fmaxf(fmaxf(x0.y, y0.y), fmaxf(z0.y, 0.0f)), fb = fminf(fminf(x1.y, y1.y), z1.y);
    h0 = !(na > kFarMargin * fa) && r0 != RT_EMPTY;
    h1 = !(nb > kFarMargin * fb) && r1 != RT_EMPTY;
}

// Two Gaussians as the rays of a shaft see them (step 2).
struct ShaftCand {
    float2 r11, r12, c1, r22, c2, qx, qy;
    float2 thr, h;  // passes unless |v|^2 >= thr or z + qx x + qy y >= h
};

// With W = S^-1 R^T (rows w_k) and f_i = S R^T e_i (= W e_i / |w_k|^2 per row),
// the covariance across d is [A B; B C] = f_i . f_j with determinant
// |W d|^2 / (|d|^2 prod |w_k|^2), so
//   m^2 = (x - (B / C) y)^2 C / det + y^2 / C
// without a difference of large terms.  t* of a ray from r is q . (mu - r),
// q = W^T W d / |W d|^2.  p = mu - c - s d is the mean moved along d next to
// the rays.
// Error bound, in ulps eps = 2^-24, for a ray that gauss_eval may accept (m the
// largest m it accepts, s_max the longest axis): every term of v is at most
// |W| (group radius + |p|), and mu - c carries |s| ulps.  f_k is off by eps
// s_k whatever its size, u by eps |w_k|, so C, B and |W d|^2 are off by up to
// a few eps s_max |W| of themselves where the projections are small (needles
// seen nearly end-on, discs edge-on), and v with them, |v| <= m: this does
// not shrink with the rays' distance.  gauss_eval's peak lies up to m s_max
// from mu, which puts eps |W| m s_max into its u.  Hence `reach`, the group
// radius + |p| + m s_max, at 40 eps; the limit of |v|^2 moves by E (2 m + E).
// The same lengths bound t*, in units of 1 / |W d|.
// frame: fr[0] = (c, |d|^2), fr[1] = (d, |d|), fr[2] = (d / |d|^2, group
// radius), fr[3] = (e1, k_sigma^2 log2(e)/2), fr[4] = (e2, log2(alpha_min)).
template <bool GRAD>
__device__ __forceinline__ void shaft_cand(const ShaftSmem<GRAD> &sm, const float4 (&a)[4], const float4 (&b)[4],
                                           ShaftCand &g) {
    const float4 F0 = sm.fr[0], F1 = sm.fr[1], F2 = sm.fr[2], F3 = sm.fr[3], F4 = sm.fr[4];
    const f2x3 w0 = pack3(a[1], b[1]), w1 = pack3(a[2], b[2]), w2 = pack3(a[3], b[3]);
    f2x3 p = pack3(a[0], b[0]);
    p.x = __fadd2_rn(p.x, dup(-F0.x));
    p.y = __fadd2_rn(p.y, dup(-F0.y));
    p.z = __fadd2_rn(p.z, dup(-F0.z));
    const float2 s = dot2(p, F2), ns = make_float2(-s.x, -s.y);
    p.x = __ffma2_rn(ns, dup(F1.x), p.x);
    p.y = __ffma2_rn(ns, dup(F1.y), p.y);
    p.z = __ffma2_rn(ns, dup(F1.z), p.z);
    const float2 px = dot2(p, F3), py = dot2(p, F4), pz = dot2(p, F2);
    const float2 u0 = dot2(w0, F1), u1 = dot2(w1, F1), u2 = dot2(w2, F1);
    const float2 a0 = dot2(w0, F3), a1 = dot2(w1, F3), a2 = dot2(w2, F3);
    const float2 b0 = dot2(w0, F4), b1 = dot2(w1, F4), b2 = dot2(w2, F4);
    const float2 n0 = dot2(w0, w0), n1 = dot2(w1, w1), n2 = dot2(w2, w2);
    auto rcp = [](float2 v) { return make_float2(__fdividef(1.0f, v.x), __fdividef(1.0f, v.y)); };
    auto rsq = [](float2 v) { return make_float2(rsqrtf(v.x), rsqrtf(v.y)); };
    auto mul = [](float2 x, float2 y) { return __fmul2_rn(x, y); };
    auto fma2 = [](float2 x, float2 y, float2 z) { return __ffma2_rn(x, y, z); };
    const float2 f0 = mul(b0, rcp(n0)), f1 = mul(b1, rcp(n1)), f2 = mul(b2, rcp(n2));
    // B uses f1_k f2_k = (a_k / n_k) f_k = a_k (f_k / n_k)
    const float2 B = fma2(mul(a0, rcp(n0)), f0, fma2(mul(a1, rcp(n1)), f1, mul(mul(a2, rcp(n2)), f2)));
    const float2 C = fma2(f0, f0, fma2(f1, f1, mul(f2, f2)));
    const float2 uu = fma2(u0, u0, fma2(u1, u1, mul(u2, u2)));
    const float2 iu = rcp(uu), iC = rcp(C), ru = rsq(uu);
    const float2 kap = dup(0.84932180f);  // sqrt(log2(e) / 2)
    const float2 r2 = mul(mul(mul(C, n0), mul(mul(n1, iu), n2)), dup(F0.w));
    g.r11 = mul(mul(kap, r2), rsq(r2));  // roots to 2 ulps: E holds many times that
    g.r22 = mul(kap, rsq(C));
    const float2 r12 = mul(mul(B, iC), g.r11);
    g.r12 = make_float2(-r12.x, -r12.y);
    const float2 c1 = fma2(g.r11, px, mul(g.r12, py)), c2 = mul(g.r22, py);
    g.c1 = make_float2(-c1.x, -c1.y);
    g.c2 = make_float2(-c2.x, -c2.y);
    g.qx = mul(fma2(u0, a0, fma2(u1, a1, mul(u2, a2))), iu);
    g.qy = mul(fma2(u0, b0, fma2(u1, b1, mul(u2, b2))), iu);
    const float2 nn = __fadd2_rn(n0, __fadd2_rn(n1, n2));
    const float2 hb = __fadd2_rn(__fadd2_rn(s, pz), fma2(g.qx, px, mul(g.qy, py)));
    auto lim = [&](float nn1, float nmin, float px1, float py1, float s1, float ru1, float o, float h1, float &thr,
                   float &h) {
        const float L = fminf(F3.w, __log2f(o) - F4.w), l = fmaxf(L, 1e-20f), m = l * rsqrtf(l);  // |v| <= m; 1.18 m sigma
        const float wn = nn1 * rsqrtf(nn1), reach = fmaf(1.18f * m, rsqrtf(nmin), F2.w + fabsf(px1) + fabsf(py1)),
                    sl = fabsf(s1) * F1.w;
        const float E = wn * fmaf(2.4e-6f, reach, 4e-7f * sl);
        thr = fmaf(E, fmaf(2.0f, m, E), fmaf(L, 1.000001f, 1e-5f));
        h = fmaf(2e-6f, fmaf(wn * (reach + sl), ru1, fabsf(s1)), h1);
    };
    const float na = fminf(n0.x, fminf(n1.x, n2.x)), nb = fminf(n0.y, fminf(n1.y, n2.y));
    lim(nn.x, na, px.x, py.x, s.x, ru.x, a[0].w, hb.x, g.thr.x, g.h.x);
    lim(nn.y, nb, px.y, py.y, s.y, ru.y, b[0].w, hb.y, g.thr.y, g.h.y);
}

// gauss_eval of two pairs at once, each operation rounded as there.
struct PairEval {
    f2x3 w0, w1, w2, hi, lo, D;
    float2 num, den, alpha;  // t* = -num / den
    bool acc[2];
    __device__ __forceinline__ float2 dot(f2x3 x, f2x3 y) const {
        return __ffma2_rn(x.x, y.x, __ffma2_rn(x.y, y.y, __fmul2_rn(x.z, y.z)));
    }
    __device__ __forceinline__ f2x3 peak(float2 t) const {  // x(t) - mu
        f2x3 e;
        e.x = __fadd2_rn(__ffma2_rn(t, D.x, hi.x), lo.x);
        e.y = __fadd2_rn(__ffma2_rn(t, D.y, hi.y), lo.y);
        e.z = __fadd2_rn(__ffma2_rn(t, D.z, hi.z), lo.z);
        return e;
    }
    __device__ __forceinline__ f2x3 whiten(f2x3 e) const {
        f2x3 u;
        u.x = dot(w0, e);
        u.y = dot(w1, e);
        u.z = dot(w2, e);
        return u;
    }
    __device__ __forceinline__ PairEval(const BvhDev &b, const float4 (&ga)[4], const float4 (&gb)[4], float4 oa,
                                        float4 ob, float3 d) {
        const f2x3 mu = pack3(ga[0], gb[0]), o = pack3(oa, ob);
        w0 = pack3(ga[1], gb[1]);
        w1 = pack3(ga[2], gb[2]);
        w2 = pack3(ga[3], gb[3]);
        two_diff2(o.x, mu.x, hi.x, lo.x);
        two_diff2(o.y, mu.y, hi.y, lo.y);
        two_diff2(o.z, mu.z, hi.z, lo.z);
        D.x = dup(d.x);
        D.y = dup(d.y);
        D.z = dup(d.z);
        const f2x3 ud = whiten(D), uo = whiten(hi);
        num = dot(uo, ud);
        den = dot(ud, ud);
        const float2 t = make_float2(__fdividef(-num.x, den.x), __fdividef(-num.y, den.y));
        const f2x3 u = whiten(peak(t));
        const float2 m2 = dot(u, u);
        alpha = make_float2(ga[0].w * __expf(-0.5f * m2.x), gb[0].w * __expf(-0.5f * m2.y));
        acc[0] = t.x > 0.0f && m2.x <= b.k2 && alpha.x >= b.alpha_min;
        acc[1] = t.y > 0.0f && m2.y <= b.k2 && alpha.y >= b.alpha_min;
    }
};

// T of the `count` (1..64) rays of sorted positions first, first + 1, ...
// along d (the same in every lane): in sm.ro[i].w, not snapped.
// GRAD: `gr` has the rays' dL/dT and T and takes their hits' gradients (rays
// without a gradient never join the group; none leaves it).
template <bool GRAD, class Grad = int>
__device__ __forceinline__ void shaft_group(const BvhDev &b, float eps, float3 d, int64_t first, int count,
                                            int *status, ShaftSmem<GRAD> &sm, Grad *gr = nullptr) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const float inf = __int_as_float(0x7f800000);
    float3 inv, oi;
    // false: the rays meet nothing (their boxes' tests, all NaN, would let every node pass)
    const bool finite = qnode_ray(make_float3(eps * d.x, eps * d.y, eps * d.z), d, inv, oi);
    int live = count;
    if constexpr (GRAD) live = 0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int i = lane + 32 * r;
        int slot = i;
        float w = 1.0f;
        bool in = i < count;
        if constexpr (GRAD) {
            w = gr->load(b, first, i, in);
            const unsigned v = __ballot_sync(FULL, in);
            slot = live + __popc(v & lt);
            live += __popc(v);
        }
        if (!in) continue;
        const float4 mu = __ldg(b.gauss + 4 * (first + i));
        sm.ro[slot] = make_float4(__fadd_rn(mu.x, __fmul_rn(eps, d.x)), __fadd_rn(mu.y, __fmul_rn(eps, d.y)),
                                  __fadd_rn(mu.z, __fmul_rn(eps, d.z)), w);
        sm.live[slot] = (uint8_t)i;
    }
    if constexpr (GRAD) {
        gr->live = live;
        if (live == 0) return;
        __syncwarp();
    }
    // the box of n live rays' origins: centre c, half extents hh (outwards)
    float3 c, hh, cn, cf;
    auto bounds = [&](int n) {
        float3 lo = make_float3(inf, inf, inf), hi = make_float3(-inf, -inf, -inf);
        for (int s = lane; s < n; s += 32) {
            const float4 o = sm.ro[GRAD ? s : sm.live[s]];
            lo = make_float3(fminf(lo.x, o.x), fminf(lo.y, o.y), fminf(lo.z, o.z));
            hi = make_float3(fmaxf(hi.x, o.x), fmaxf(hi.y, o.y), fmaxf(hi.z, o.z));
        }
        lo = make_float3(warp_min(lo.x), warp_min(lo.y), warp_min(lo.z));
        hi = make_float3(warp_max(hi.x), warp_max(hi.y), warp_max(hi.z));
        c = make_float3(0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y), 0.5f * (lo.z + hi.z));
        hh = make_float3(1.000001f * fmaxf(hi.x - c.x, c.x - lo.x), 1.000001f * fmaxf(hi.y - c.y, c.y - lo.y),
                         1.000001f * fmaxf(hi.z - c.z, c.z - lo.z));
        const float3 w = make_float3(hh.x * fabsf(inv.x), hh.y * fabsf(inv.y), hh.z * fabsf(inv.z));
        cn = make_float3(fmaf(c.x, inv.x, w.x), fmaf(c.y, inv.y, w.y), fmaf(c.z, inv.z, w.z));
        cf = make_float3(fmaf(c.x, inv.x, -w.x), fmaf(c.y, inv.y, -w.y), fmaf(c.z, inv.z, -w.z));
    };
    bounds(live);
    {
        // plane frame (e1, e2) across d (Duff et al. 2017); d scaled by a power
        // of two (exact) to a largest component in [1, 2): |d|^2 is in range, and
        // all that the rejection test computes is in units of |d|
        const uint32_t e = __float_as_uint(fmaxf(fmaxf(fabsf(d.x), fabsf(d.y)), fabsf(d.z))) >> 23;
        const float pw = __uint_as_float((e < 253u ? 254u - e : 1u) << 23);
        const float3 ds = make_float3(d.x * pw, d.y * pw, d.z * pw);
        const float dd = dot3(ds, ds), il = rsqrtf(dd);
        const float3 dn = make_float3(ds.x / dd, ds.y / dd, ds.z / dd);
        const float x = ds.x * il, y = ds.y * il, z = ds.z * il;
        const float sg = copysignf(1.0f, z), a = -1.0f / (sg + z), q = x * y * a;
        const float3 e1 = make_float3(1.0f + sg * x * x * a, sg * q, -sg * x), e2 = make_float3(q, sg + y * y * a, -y);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int i = lane + 32 * r;
            if (i >= live) continue;
            const float4 o = sm.ro[i];
            const float3 v = make_float3(o.x - c.x, o.y - c.y, o.z - c.z);
            sm.xy[i] = make_float2(dot3(e1, v), dot3(e2, v));
            sm.z[i] = dot3(dn, v);
        }
        if (lane == 0) {
            sm.fr[0] = make_float4(c.x, c.y, c.z, dd);
            sm.fr[1] = make_float4(ds.x, ds.y, ds.z, sqrtf(dd));
            sm.fr[2] = make_float4(dn.x, dn.y, dn.z, hh.x + hh.y + hh.z);
            sm.fr[3] = make_float4(e1.x, e1.y, e1.z, 0.72134752f * b.k2);
            sm.fr[4] = make_float4(e2.x, e2.y, e2.z, log2f(b.alpha_min));
            sm.stack[0] = 0u;
        }
    }
    // step 2: 16-byte row r of staged record i lies at chunk r ^ ((i >> 1) & 3)
    auto rec = [&](int i, int r) { return sm.stage[4 * i + (r ^ ((i >> 1) & 3))]; };
    const int room = kShaftStack - 4 - 3 * b.levels;  // beyond it, nodes are walked one at a time
    int bound = live, size = finite ? 1 : 0, nleaf = 0;
    (void)bound;
    __syncwarp();
    for (;;) {
        while (nleaf < kShaftCands && size > 0) {
            const int k = min(min(kShaftNodes, size), min(max(1, (room - size) / 3), (kShaftLeaves - nleaf) / 4));
            size -= k;
            const uint32_t node = (lane >> 1) < k ? sm.stack[size + (lane >> 1)] : 0u;
            __syncwarp();
            bool h0 = false, h1 = false;
            uint32_t r0 = 0u, r1 = 0u;
            if ((lane >> 1) < k) shaft_qnode(b.qwide + 4 * (int64_t)node, lane & 1, inv, cn, cf, h0, h1, r0, r1);
            const bool f0 = h0 && (int)r0 < 0, f1 = h1 && (int)r1 < 0;
            h0 = h0 && !f0;
            h1 = h1 && !f1;
            const unsigned bf0 = __ballot_sync(FULL, f0), bf1 = __ballot_sync(FULL, f1);
            const unsigned bh0 = __ballot_sync(FULL, h0), bh1 = __ballot_sync(FULL, h1);
            if (f0) sm.leaf[nleaf + __popc(bf0 & lt)] = r0 & ~RT_LEAF_BIT;
            nleaf += __popc(bf0);
            if (f1) sm.leaf[nleaf + __popc(bf1 & lt)] = r1 & ~RT_LEAF_BIT;
            nleaf += __popc(bf1);
            if (h0) sm.stack[size + __popc(bh0 & lt)] = r0;
            size += __popc(bh0);
            if (h1) sm.stack[size + __popc(bh1 & lt)] = r1;
            size += __popc(bh1);
            __syncwarp();
            if (size > kShaftStack - 4) {  // never: 3 a level beyond `room`
                if (lane == 0) rt_set_error(status, RT_ERR_STACK_OVERFLOW);
                size = 0;
            }
        }
        if (nleaf == 0) break;
        const int m = min(kShaftCands, nleaf);
        nleaf -= m;
        // 64-byte records by 4 lanes each
#pragma unroll
        for (int t = 0; t < kShaftCands / 8; ++t) {
            const int i = 8 * t + (lane >> 2);
            if (i < m)
                cp_async16(sm.stage + 4 * i + ((lane ^ (i >> 1)) & 3), b.gauss + 4 * (int64_t)sm.leaf[nleaf + i] + (lane & 3));
        }
        cp_async_done();
        __syncwarp();
        ShaftCand g;
        {
            // lanes past the batch repeat its first Gaussian (their votes are dropped)
            const int ia = lane < m ? lane : 0, ib = lane + 32 < m ? lane + 32 : 0;
            const float4 ra[4] = {rec(ia, 0), rec(ia, 1), rec(ia, 2), rec(ia, 3)};
            const float4 rb[4] = {rec(ib, 0), rec(ib, 1), rec(ib, 2), rec(ib, 3)};
            shaft_cand(sm, ra, rb, g);
        }
        uint2 ca = make_uint2(0u, 0u), cb = ca;  // GRAD: the slots that voted for this lane's Gaussians
#pragma unroll 2
        for (int t = 0; t < live; ++t) {
            const float2 v = sm.xy[t], X = dup(v.x), Y = dup(v.y);
            const float2 v1 = __ffma2_rn(g.r11, X, __ffma2_rn(g.r12, Y, g.c1)), v2 = __ffma2_rn(g.r22, Y, g.c2);
            const float2 q = __ffma2_rn(v1, v1, __fmul2_rn(v2, v2));
            const float2 z = __ffma2_rn(g.qx, X, __ffma2_rn(g.qy, Y, dup(sm.z[t])));
            const bool pa = !(q.x >= g.thr.x) && !(z.x >= g.h.x), pb = !(q.y >= g.thr.y) && !(z.y >= g.h.y);
            const uint32_t ma = __ballot_sync(FULL, pa), mb = __ballot_sync(FULL, pb);
            if (lane == 0) sm.mask[t] = make_uint2(ma, mb);
            if constexpr (GRAD) {
                const uint32_t bit = 1u << (t & 31), b0 = t < 32 ? bit : 0u, b1 = t < 32 ? 0u : bit;
                ca.x |= pa ? b0 : 0u;
                ca.y |= pa ? b1 : 0u;
                cb.x |= pb ? b0 : 0u;
                cb.y |= pb ? b1 : 0u;
            }
        }
        __syncwarp();
        if constexpr (GRAD) {
            if (lane >= m) ca = make_uint2(0u, 0u);
            if (lane + 32 >= m) cb = make_uint2(0u, 0u);
            gr->batch(b, d, first, live, m, sm.leaf + nleaf, ca, cb, sm);
        } else {
            // step 3, the live rays of 32 slots at a time
            for (int s0 = 0; s0 < live; s0 += 32) {
                uint2 mk = make_uint2(0u, 0u);
                uint32_t ray = 0u;
                if (s0 + lane < live) {
                    mk = sm.mask[s0 + lane];
                    // a NaN test passes: not in the lanes past the batch
                    mk.x &= m >= 32 ? FULL : (1u << m) - 1u;
                    mk.y &= m >= 64 ? FULL : m > 32 ? (1u << (m - 32)) - 1u : 0u;
                    ray = sm.live[s0 + lane];
                }
                while (__any_sync(FULL, (mk.x | mk.y) != 0u)) {
                    int na = __popc(mk.x), nb = __popc(mk.y);
                    if (__reduce_add_sync(FULL, na + nb) > kShaftPairs<GRAD>) {  // a part of each ray's
                        na = min(na, kShaftPairs<GRAD> / 64);
                        nb = min(nb, kShaftPairs<GRAD> / 64);
                    }
                    int end = na + nb;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int v = __shfl_up_sync(FULL, end, off);
                        if (lane >= off) end += v;
                    }
                    const int total = __shfl_sync(FULL, end, 31), from = end - na - nb;
                    int at = from;
                    for (; na > 0; --na) {
                        sm.pair[at++] = ray << 6 | (uint32_t)(__ffs(mk.x) - 1);
                        mk.x &= mk.x - 1u;
                    }
                    for (; nb > 0; --nb) {
                        sm.pair[at++] = ray << 6 | (uint32_t)(__ffs(mk.y) + 31);
                        mk.y &= mk.y - 1u;
                    }
                    __syncwarp();
                    for (int i = lane; i < total; i += 64) {
                        const uint32_t pa = sm.pair[i], pb = i + 32 < total ? sm.pair[i + 32] : pa;
                        const int qa = pa & 63u, qb = pb & 63u;
                        const float4 oa = sm.ro[pa >> 6], ob = sm.ro[pb >> 6];
                        const float4 ra[4] = {rec(qa, 0), rec(qa, 1), rec(qa, 2), rec(qa, 3)};
                        const float4 rb[4] = {rec(qb, 0), rec(qb, 1), rec(qb, 2), rec(qb, 3)};
                        const PairEval e(b, ra, rb, oa, ob, d);
                        float fa = e.acc[0] ? 1.0f - e.alpha.x : 1.0f, fb = e.acc[1] ? 1.0f - e.alpha.y : 1.0f;
                        if (sm.leaf[nleaf + qa] == (uint32_t)first + (pa >> 6)) fa = 1.0f;  // the ray's own Gaussian
                        if (sm.leaf[nleaf + qb] == (uint32_t)first + (pb >> 6)) fb = 1.0f;
                        sm.pair[i] = __float_as_uint(fa);
                        if (i + 32 < total) sm.pair[i + 32] = __float_as_uint(fb);
                    }
                    __syncwarp();
                    if (s0 + lane < live) {
                        float T = sm.ro[ray].w;
                        for (int i = from; i < end; ++i) T *= __uint_as_float(sm.pair[i]);
                        sm.ro[ray].w = T;
                        if (T < b.t_min) mk = make_uint2(0u, 0u);
                    }
                    __syncwarp();
                }
            }
            // the rays still live, closed up
            bool ok[2];
            float2 vxy[2];
            float vz[2];
            uint8_t id[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int s = lane + 32 * r;
                ok[r] = s < live;
                if (ok[r]) {
                    id[r] = sm.live[s];
                    ok[r] = !(sm.ro[id[r]].w < b.t_min);
                }
            }
            const unsigned k0 = __ballot_sync(FULL, ok[0]), k1 = __ballot_sync(FULL, ok[1]);
            const int now = __popc(k0) + __popc(k1);
            if (now == 0) break;
            if (now < live) {
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    if (ok[r]) {
                        vxy[r] = sm.xy[lane + 32 * r];
                        vz[r] = sm.z[lane + 32 * r];
                    }
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    if (ok[r]) {
                        const int s = r == 0 ? __popc(k0 & lt) : __popc(k0) + __popc(k1 & lt);
                        sm.xy[s] = vxy[r];
                        sm.z[s] = vz[r];
                        sm.live[s] = id[r];
                    }
                live = now;
                if (4 * live <= 3 * bound) {  // the shaft of the rays left
                    bound = live;
                    __syncwarp();
                    bounds(live);
                }
            }
        }
        __syncwarp();
    }
    __syncwarp();
}

// One item of a direction set: group and direction, T written in the caller's
// order.
__device__ __forceinline__ void shaft_item(const BvhDev &b, const RaySetDev &rs, const TraceJob &job, float *T_out,
                                           int64_t item, int *status, ShaftSmem<false> &sm) {
    int64_t gi;
    int32_t k;
    full_item(job, rs.K, item, gi, k);
    const int2 gr = __ldg(b.groups + gi);
    shaft_group<false>(b, rs.eps, make_float3(__ldg(rs.dirs + 3 * k), __ldg(rs.dirs + 3 * k + 1), __ldg(rs.dirs + 3 * k + 2)),
                gr.x, gr.y, status, sm);
    for (int i = threadIdx.x & 31; i < gr.y; i += 32) {
        const int64_t g = __float_as_int(__ldg(b.gauss + 4 * (int64_t)(gr.x + i) + 1).w);
        const float T = sm.ro[i].w;
        T_out[g * rs.K + k] = T < b.t_min ? 0.0f : T;
    }
    __syncwarp();
}

// Resident blocks of 128 threads per SM: 37 KB of shared memory each.
constexpr int kShaftBlocks = 6;
