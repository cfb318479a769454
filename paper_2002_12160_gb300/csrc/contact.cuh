// contact.cuh -- per-contact device arithmetic shared by the forward step
// (step_kernel.cuh, step_pd.cu) and its adjoint (adjoint.cu): narrowphase of a sphere against the
// palm box and a finger capsule, the contact's bias and effective masses, one
// projected Jacobi update, and the 6-value sum over the lanes of a group.
// The kernels include this header so that the adjoint differentiates the expressions
// the step runs; outside it their forwards differ in which product of a few sums is
// rounded first (internal.cuh, prod_add), that is by rounding alone.
#pragma once

#include "internal.cuh"

namespace ih {

struct Hit {
    float gap;
    V3 n;     // from the link toward the object
    float t;  // axial fraction along a capsule, 0 on the palm
};

// sphere (centre c, radius rs) against a box of the given half extents at the
// origin of c's frame
__device__ __forceinline__ Hit hit_box_local(V3 c, float rs, float hx, float hy, float hz) {
    const V3 k = mk(fminf(fmaxf(c.x, -hx), hx), fminf(fmaxf(c.y, -hy), hy), fminf(fmaxf(c.z, -hz), hz));
    Hit h;
    h.t = 0.0f;
    const bool inside = (k.x == c.x) && (k.y == c.y) && (k.z == c.z);
    if (!inside) {
        const V3 d = c - k;
        const float d2 = dot(d, d);
        const float inv = rsqrtf(d2);   // d2 > 0: the centre is outside the box
        h.n = d * inv;
        h.gap = d2 * inv - rs;
    } else {
        // shallowest face, ties to the lowest axis and the + side
        float best = hx - c.x;
        h.n = mk(1, 0, 0);
        if (hx + c.x < best) { best = hx + c.x; h.n = mk(-1, 0, 0); }
        if (hy - c.y < best) { best = hy - c.y; h.n = mk(0, 1, 0); }
        if (hy + c.y < best) { best = hy + c.y; h.n = mk(0, -1, 0); }
        if (hz - c.z < best) { best = hz - c.z; h.n = mk(0, 0, 1); }
        if (hz + c.z < best) { best = hz + c.z; h.n = mk(0, 0, -1); }
        h.gap = -best - rs;
    }
    return h;
}

// sphere at ca (relative to the capsule start) against the axis s d, s in [0, L]
__device__ __forceinline__ Hit hit_capsule(V3 ca, float rs, V3 d, float L, float inv_L, float rc, Q4 q) {
    const float t = fminf(fmaxf(dot(ca, d) * inv_L, 0.0f), 1.0f);
    const V3 diff = ca - d * (t * L);
    const float d2 = dot(diff, diff);
    Hit h;
    h.t = t;
    if (d2 < 1e-18f) {   // centre on the axis
        h.n = qrot(q, mk(0, 0, 1));
        h.gap = -rs - rc;
    } else {
        const float inv = rsqrtf(d2);
        h.n = diff * inv;
        h.gap = d2 * inv - rs - rc;
    }
    return h;
}

constexpr int kMaxLinks = 32;
constexpr int kSphStride = kCluster + 1;   // spheres of a cluster, padded: lanes on different clusters hit different banks
// Centre of the spheres that fill a shape's last cluster: its squared distance from
// anything overflows, so that no margin, however large, makes them contacts
constexpr float kFar = 3e38f;

// Per link its pads in order and their intervals [s0, s1) (absent: an interval
// that holds nothing; the palm: its first pad holds all).
struct alignas(16) PadTable {
    static constexpr int kPerLink = 4;
    float s0[kMaxLinks][kPerLink], s1[kMaxLinks][kPerLink];
    unsigned char id[kMaxLinks][kPerLink];
    __device__ void build(const DevScene &sc, int first, int step) {
#pragma unroll 1
        for (int l = first; l < sc.n_links; l += step) {
            int c = 0;
#pragma unroll 1
            for (int p = 0; p < sc.n_pads && c < (l == 0 ? 1 : kPerLink); ++p) {
                if (__ldg(sc.pad_link + p) != l) continue;
                const float e = __ldg(sc.pad_s1 + p);
                s0[l][c] = l == 0 ? -1.0f : __ldg(sc.pad_s0 + p);
                s1[l][c] = (l == 0 || e >= 1.0f) ? 2.0f : e;   // (t <= 1)
                id[l][c++] = (unsigned char)p;
            }
#pragma unroll 1
            for (; c < kPerLink; ++c) {
                s0[l][c] = 3.0f;
                s1[l][c] = 3.0f;
                id[l][c] = 0xff;
            }
        }
    }
    // the first pad of link l whose interval holds t (0xff: none)
    __device__ __forceinline__ unsigned char find(int l, float t) const {
        const float4 b = *reinterpret_cast<const float4 *>(s0[l]), e = *reinterpret_cast<const float4 *>(s1[l]);
        const uchar4 i = *reinterpret_cast<const uchar4 *>(id[l]);
        unsigned char pad = 0xff;
        if (t >= b.w && t < e.w) pad = i.w;
        if (t >= b.z && t < e.z) pad = i.z;
        if (t >= b.y && t < e.y) pad = i.y;
        if (t >= b.x && t < e.x) pad = i.x;
        return pad;
    }
};

// from the palm box (its pose is the identity, fk_kernel) to a point
__device__ __forceinline__ V3 palm_offset(const DevScene &sc, V3 c) {
    return c - mk(fminf(fmaxf(c.x, -sc.palm_hx), sc.palm_hx), fminf(fmaxf(c.y, -sc.palm_hy), sc.palm_hy),
                  fminf(fmaxf(c.z, -sc.palm_hz), sc.palm_hz));
}

// Whether a cluster's enclosing sphere (centre ca from link l's origin, radius rs)
// reaches the link, ld its axis; a little wider than it need be: the sphere tests decide
__device__ __forceinline__ bool cluster_reaches(const DevScene &sc, const DevConfig &cfg, int l, V3 ca, float rs, V3 ld) {
    const V3 dc = ca - ld * fminf(fmaxf(dot(ca, ld), 0.0f), sc.link_len), dp = palm_offset(sc, ca);
    const V3 dd = l == 0 ? dp : dc;
    const float reach = (rs + cfg.margin + (l == 0 ? 0.0f : sc.link_rad)) * 1.00001f;
    return dot(dd, dd) < reach * reach;
}

// Whether a sphere's gap to link l is below the margin, in the contact setup's own
// arithmetic (the rare pairs that the squared distance leaves open; out of line)
static __device__ __noinline__ bool gap_below_margin(const DevScene &sc, float margin, int l, V3 ca, float rs, V3 ld) {
    const Hit h = l == 0 ? hit_box_local(ca, rs, sc.palm_hx, sc.palm_hy, sc.palm_hz)
                         : hit_capsule(ca, rs, ld, sc.link_len, 1.0f / sc.link_len, sc.link_rad, {1.0f, 0.0f, 0.0f, 0.0f});
    return h.gap < margin;   // (the gap does not depend on the link's rotation)
}

// The contacts (bit i: sphere i) among the eight spheres sk of cluster k against
// link l (xa: the object's origin from the link's). A sphere is a contact when its
// gap is below the margin, which its squared distance from the link's axis (or
// box) decides unless it is within 1e-5 of the reach squared (the gap's rounding,
// rsqrtf's two ulp above all, moves the squared distance by less than a tenth of
// that): those are tested again by their gap.
__device__ __forceinline__ unsigned cluster_hits(const DevScene &sc, const DevConfig &cfg, int l, int k, V3 xa, V3 ld,
                                                 const float4 *sk, int NS, float inv_L) {
    unsigned hits = 0, close = 0;
    auto mark = [&](V3 dd, float reach, int i) {
        const float d2 = dot(dd, dd), r2 = reach * reach, over = d2 - r2;
        if (over < 0.0f) hits |= 1u << i;
        if (!(fabsf(over) > 1e-5f * r2)) close |= 1u << i;
    };
    if (l == 0) {
#pragma unroll
        for (int i = 0; i < kCluster; ++i) {
            const float4 c4 = sk[i];
            mark(palm_offset(sc, xa + xyz(c4)), c4.w + cfg.margin, i);
        }
    } else {
        const float rm = sc.link_rad + cfg.margin;
#pragma unroll
        for (int i = 0; i < kCluster; ++i) {
            const float4 c4 = sk[i];
            const V3 ca = xa + xyz(c4);
            const float t = fminf(fmaxf(dot(ca, ld) * inv_L, 0.0f), 1.0f);
            mark(ca - ld * (t * sc.link_len), c4.w + rm, i);
        }
    }
#pragma unroll 1
    for (; close; close &= close - 1u) {   // rare
        const int i = __ffs(close) - 1;
        const float4 c4 = sk[i];
        const bool hit = k * kCluster + i < NS && gap_below_margin(sc, cfg.margin, l, xa + xyz(c4), c4.w, ld);
        hits = (hits & ~(1u << i)) | (hit ? 1u << i : 0u);
    }
    return hits;
}

// A sphere of the object (centre cr from the object's origin) against link l: its hit
__device__ __forceinline__ Hit hit_link(const DevScene &sc, int l, V3 ca, float rs, V3 ld, const float4 *L0, float inv_L) {
    if (l == 0) return hit_box_local(ca, rs, sc.palm_hx, sc.palm_hy, sc.palm_hz);
    const float4 q = __ldg(L0 + l * kLinkStride + 2);
    return hit_capsule(ca, rs, ld, sc.link_len, inv_L, sc.link_rad, {q.x, q.y, q.z, q.w});
}

// (one division for both regimes, so that a warp that mixes them divides once)
__device__ __forceinline__ float contact_bias(const DevConfig &cfg, float gap) {
    const float q = (gap > 0.0f ? gap : cfg.beta * fminf(gap + cfg.slop, 0.0f)) / cfg.h;
    return gap > 0.0f ? q : fmaxf(q, -cfg.vmax);
}

__device__ __forceinline__ bool all_finite(V3 x, Q4 q, V3 v, V3 w) {
    return isfinite(x.x) && isfinite(x.y) && isfinite(x.z) && isfinite(q.w) && isfinite(q.x) &&
           isfinite(q.y) && isfinite(q.z) && isfinite(v.x) && isfinite(v.y) && isfinite(v.z) &&
           isfinite(w.x) && isfinite(w.y) && isfinite(w.z);
}

// Per-contact constants: scalar effective masses along the normal and in the
// tangent plane, and the target velocity c = v_link - b n (bias folded in).
struct CSetup {
    float ikn, ikt;
    V3 cc;
};

__device__ __forceinline__ CSetup setup_contact(V3 r, V3 n, float gap, int l, const S6 &Wi, float trW, float inv_m,
                                                const DevConfig &cfg, const float4 *L0, const float4 *L1, V3 x,
                                                float inv_h) {
    // k_n = 1/m + (r x n)^T W (r x n); tr K = 3/m + |r|^2 tr W - r^T W r
    const V3 rn = cross(r, n);
    const float kn = inv_m + dot(rn, smul(Wi, rn));
    const float trK = prod_add(3.0f, inv_m, dot(r, r), trW) - dot(r, smul(Wi, r));
    CSetup c;
    c.ikn = 1.0f / kn;
    c.ikt = 2.0f / (trK - kn);
    const float b = contact_bias(cfg, gap);
    V3 vl = mk(0, 0, 0);
    if (l != 0) {   // link point velocity from the link's rigid displacement over the substep
        const float4 A0 = __ldg(L0 + l * kLinkStride), B0 = __ldg(L1 + l * kLinkStride);
        const float4 Aq = __ldg(L0 + l * kLinkStride + 2), Bq = __ldg(L1 + l * kLinkStride + 2);
        const Q4 qa = {Aq.x, Aq.y, Aq.z, Aq.w}, qb = {Bq.x, Bq.y, Bq.z, Bq.w};
        const V3 pl = qrot_inv(qa, (x - xyz(A0)) + r);   // contact in link coords
        const V3 d = (xyz(B0) - xyz(A0)) + (qrot(qb, pl) - qrot(qa, pl));
        vl = {__fmul_rn(d.x, inv_h), __fmul_rn(d.y, inv_h), __fmul_rn(d.z, inv_h)};
    }
    c.cc = vl - n * b;
    return c;
}

// One projected Jacobi update of a contact's impulse lam against the body velocity
// (v, w): scalar normal step clamped at zero, scalar tangential step clamped
// radially to the Coulomb disk, relaxed by 1/n_c:
//   u = v + w x r - c,  l_n = max(lam . n - (u . n) / k_n, 0),
//   l_t = (lam - n (lam . n)) - (u - n (u . n)) / k_t, scaled to mu l_n where longer,
//   lam += (n l_n + l_t - lam) / n_c,
// with a fixed contraction. The disk clamp is a select, not a branch, so that the
// sliding and the sticking lanes of a warp stay in one stretch of code. On one
// contact (T = float) or on two at once (T = float2, the packed FP32 instructions:
// half the issue slots of two scalar updates, and two chains that interleave): every
// operation is the scalar one of each half. Two contacts cost ~70 issue slots instead of ~130; an iteration
// of a 60-contact environment at 16 warps per SM took 258 cycles a warp scalar,
// 198 packed. The reciprocal square root is taken of the argument scaled by
// 2^24, which no FP32 value leaves denormal, so the approximate instruction
// needs no denormal path (18 cycles instead of 40); for arguments below 2^104 it
// equals rsqrtf bit for bit (all of them compared), that is for impulses below
// 4.5e15 N s, beyond which the clamp's squares overflow (unscaled at 1.8e19).
typedef float2 F2;
__device__ __forceinline__ float t_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ F2 t_fma(F2 a, F2 b, F2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float t_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ F2 t_mul(F2 a, F2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float t_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ F2 t_add(F2 a, F2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float t_neg(float a) { return -a; }
__device__ __forceinline__ F2 t_neg(F2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float t_relu(float a) { return fmaxf(a, 0.0f); }
__device__ __forceinline__ F2 t_relu(F2 a) { return make_float2(fmaxf(a.x, 0.0f), fmaxf(a.y, 0.0f)); }
template <typename T> __device__ __forceinline__ T t_all(float a);
template <> __device__ __forceinline__ float t_all<float>(float a) { return a; }
template <> __device__ __forceinline__ F2 t_all<F2>(float a) { return make_float2(a, a); }
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// scale of the disk clamp: lim / |t| where |t| > lim, else 1, from t2 = 2^24 |t|^2 and lim = 2^12 mu l_n
__device__ __forceinline__ float t_clamp(float t2, float lim) {
    const float sc = lim * rsqrt_ftz(t2);
    return t2 > lim * lim ? sc : 1.0f;
}
__device__ __forceinline__ F2 t_clamp(F2 t2, F2 lim) { return make_float2(t_clamp(t2.x, lim.x), t_clamp(t2.y, lim.y)); }

template <typename T>
struct Vec {
    T x, y, z;
};
template <typename T>
__device__ __forceinline__ T t_dot(const Vec<T> &a, const Vec<T> &b) { return t_fma(a.x, b.x, t_fma(a.y, b.y, t_mul(a.z, b.z))); }
template <typename T>
struct Contact {
    Vec<T> r, n, c, lam;
    T ikn, ikt;
    __device__ __forceinline__ void clear() {   // an empty slot: keeps a zero impulse and adds zeros
        const T o = t_all<T>(0.0f);
        r = c = lam = {o, o, o};
        n = {o, o, t_all<T>(1.0f)};
        ikn = ikt = o;
    }
    // lam after one update against the velocity (v, w); mu_s = 2^12 mu
    __device__ __forceinline__ void update(V3 v, V3 w, float mu_s, float inv_nc) {
        const Vec<T> nv = {t_all<T>(-v.x), t_all<T>(-v.y), t_all<T>(-v.z)}, pw = {t_all<T>(w.x), t_all<T>(w.y), t_all<T>(w.z)},
                     nw = {t_all<T>(-w.x), t_all<T>(-w.y), t_all<T>(-w.z)};
        // -u = c - (v + w x r)
        const Vec<T> nu = {t_add(t_add(nv.x, t_fma(nw.y, r.z, t_mul(pw.z, r.y))), c.x),
                           t_add(t_add(nv.y, t_fma(nw.z, r.x, t_mul(pw.x, r.z))), c.y),
                           t_add(t_add(nv.z, t_fma(nw.x, r.y, t_mul(pw.y, r.x))), c.z)};
        const T nun = t_dot(nu, n), lo = t_dot(lam, n), un = t_neg(nun), nlo = t_neg(lo);
        const T ln = t_relu(t_fma(nun, ikn, lo));
        const Vec<T> t = {t_fma(t_fma(n.x, un, nu.x), ikt, t_fma(n.x, nlo, lam.x)),
                          t_fma(t_fma(n.y, un, nu.y), ikt, t_fma(n.y, nlo, lam.y)),
                          t_fma(t_fma(n.z, un, nu.z), ikt, t_fma(n.z, nlo, lam.z))};
        const T f = t_clamp(t_mul(t_dot(t, t), t_all<T>(16777216.0f)), t_mul(t_all<T>(mu_s), ln));
        const T m1 = t_all<T>(-1.0f), k = t_all<T>(inv_nc);
        lam.x = t_fma(t_fma(lam.x, m1, t_fma(n.x, ln, t_mul(t.x, f))), k, lam.x);
        lam.y = t_fma(t_fma(lam.y, m1, t_fma(n.y, ln, t_mul(t.y, f))), k, lam.y);
        lam.z = t_fma(t_fma(lam.z, m1, t_fma(n.z, ln, t_mul(t.z, f))), k, lam.z);
    }
    // its impulse and moment r x lam
    __device__ __forceinline__ void wrench(T (&s)[6]) const {
        const Vec<T> nl = {t_neg(lam.x), t_neg(lam.y), t_neg(lam.z)};
        s[0] = lam.x; s[1] = lam.y; s[2] = lam.z;
        s[3] = t_fma(r.y, lam.z, t_mul(r.z, nl.y));
        s[4] = t_fma(r.z, lam.x, t_mul(r.x, nl.z));
        s[5] = t_fma(r.x, lam.y, t_mul(r.y, nl.x));
    }
};

// Sum of 6 values over the WIDTH lanes of a group (WIDTH = 16 or 32), every
// lane receiving all 6 sums. Reduce-scatter first: padded to 8 values, each
// of the first three xor levels halves the values a lane keeps (the partner
// sends the half the lane keeps and keeps the other half), the remaining levels
// are plain; the lane at position (k>>2) W/2 + ((k>>1)&1) W/4 + (k&1) W/8
// then holds the full sum of value k, and six shuffles broadcast them.
// 15 shuffles and 9 additions for WIDTH = 32 instead of 30 and 30.
template <int WIDTH>
__device__ __forceinline__ float width_scatter6(const float (&v)[6], unsigned mask, int lane_in_group) {
    const bool b2 = lane_in_group & (WIDTH / 2), b4 = lane_in_group & (WIDTH / 4), b8 = lane_in_group & (WIDTH / 8);
    float a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float lo = v[i], hi = (i + 4 < 6) ? v[i + 4] : 0.0f;
        const float send = b2 ? lo : hi;
        a[i] = (b2 ? hi : lo) + __shfl_xor_sync(mask, send, WIDTH / 2, WIDTH);
    }
    float b[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float send = b4 ? a[i] : a[i + 2];
        b[i] = (b4 ? a[i + 2] : a[i]) + __shfl_xor_sync(mask, send, WIDTH / 4, WIDTH);
    }
    float c = (b8 ? b[1] : b[0]) + __shfl_xor_sync(mask, b8 ? b[0] : b[1], WIDTH / 8, WIDTH);
#pragma unroll
    for (int o = WIDTH / 16; o > 0; o >>= 1) c += __shfl_xor_sync(mask, c, o, WIDTH);
    return c;
}
// lane of a group holding value k after width_scatter6
template <int WIDTH>
__device__ __forceinline__ int scatter_lane(int k) {
    return (k >> 2) * (WIDTH / 2) + ((k >> 1) & 1) * (WIDTH / 4) + (k & 1) * (WIDTH / 8);
}

template <int WIDTH>
__device__ __forceinline__ void width_sum6(float (&v)[6], unsigned mask, int lane_in_group) {
    const float c = width_scatter6<WIDTH>(v, mask, lane_in_group);
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = __shfl_sync(mask, c, scatter_lane<WIDTH>(k), WIDTH);
}

}  // namespace ih
