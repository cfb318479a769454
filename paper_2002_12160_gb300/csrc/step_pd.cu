// step_pd.cu -- the dynamics step with a PD-driven articulated hand: the
// hand's joint angles are part of each environment's state (Sec. III-A, s_t
// holds the joint angles of articulated bodies) and follow the desired joint
// positions u_t through a joint-angle PD controller (Sec. IV), pushed back by
// the contacts. Each environment also reports the full observation o_t: the
// joint angles q_t, every pad's pose (P_t, R_t), its force c_t, and its
// translational slip direction d_t and rotational slip r_t (Sec. III-A).
//
// A block of one warp owns one environment (LPT order). Per substep the warp
//   1. runs the fingers' kinematics from the environment's own joint angles
//      (a lane per joint: its sine and cosine, then the finger's chain, redundantly)
//      into shared memory, with every joint's axis and origin, and predicts the
//      joints' velocities under the PD force alone:
//      qd* = (I qd + h kp (u - q)) / M, M = I + h kd + h^2 kp (implicit PD);
//   2. culls (link, 8-sphere cluster) pairs by the clusters' enclosing spheres; one
//      lane then tests the eight spheres of a surviving pair, and the contacts are
//      listed in pair order (link, then sphere);
//   3. sets each contact up: effective masses gain the joints' share
//      sum_a (J_a . n)^2 / M, J_a = z_a x (p - o_a) over the joints that move
//      the contact's link;
//   4. runs the Jacobi iterations on the object and the joints together (the
//      first 128 contacts held in registers, up to four per lane, in packed
//      pairs): each contact updates against the object velocity and its link's
//      velocity (link twist w_l x p + c_l from the joints) and leaves its impulse and
//      moment about the origin in shared memory; the warp sums the object's impulse
//      and moment, the lanes of each joint sum those of the link it ends at (with at
//      most 16 joints, one lane the forces and one the moments), a suffix over the
//      finger's lanes gives qd_a = qd*_a - z_a . sum_{links moved by a}
//      (T_l - o_a x F_l) / M, and a prefix over them the links' new twists;
//   5. integrates the object and the joints (q += h qd), and adds each
//      contact's impulse to its pad, with the impulse-weighted relative slip
//      velocity, normal and spin for the slip sensing.
// At the end of a frame the fingers' kinematics at the final joint angles give
// the pads' poses, and the slip sums give d_t and r_t. A window launch (T
// frames) writes every frame's observation, status and pose; the frames' full
// cost and window means are then formed by launches of their own (cost.cu),
// so this kernel does no FP64 work.
//
// It is bound by the latency of an iteration's chain: the contacts' updates, the links'
// sums, 16 shuffles for the joints and 15 for the object, and two passes through
// shared memory. Hence one warp a block (environments spread evenly over the SMs, the
// next starts when one ends), no branches within an iteration (one loop per number of
// occupied slots; every load of a unit before any unit's stores, 498 instead of 532
// us), a link's first eight contacts summed without a loop (357 instead of 391 us
// where an SM has one environment), and the registers of eight environments an SM
// (more of them an SM, with fewer registers: 523 us at eight, 553 at twelve, 631 at
// sixteen). Ten frames by sim_step against four-warp blocks with guarded scalar slots
// and one pair test a lane: 1024 cylinders 760 -> 492 us, 37 of them 637 -> 361 us, 64
// boxes 352 -> 248 us; 600 of mixed shapes, six frames, 722 -> 522 us.
//
// The order of every sum is fixed: lane t adds contacts t, t + 32, ... of the object's
// sums; a link's contacts are summed in order, with at most 16 joints the even and
// the odd ones apart.
#include <cstddef>

#include "contact.cuh"
#include "internal.cuh"

namespace ih {
namespace {

constexpr int kPdMaxLinks = 1 + 4 * IH_MAX_FINGERS;
constexpr int kPdMaxJoints = 4 * IH_MAX_FINGERS;
constexpr int kPdSlots = 4;                   // register-resident contacts per lane
constexpr int kPdHead = 8;                    // of a link's contacts, summed without a loop
constexpr unsigned kWarp = 0xffffffffu;
static_assert(kPdMaxLinks <= kMaxLinks && kPdMaxLinks <= 32 && kPdMaxJoints <= 32, "a lane per link and per joint");

// an environment's shared memory; the contacts' records and the centres follow
struct PdSm {
    PadTable pads;
    float4 link[kPdMaxLinks][kLinkStride];    // link poses: (a, 0), (axis, 0), (quat)
    float4 zax[kPdMaxJoints], org[kPdMaxJoints];
    float tw[6][32];                          // link twists: w_l, c_l (v(p) = w_l x p + c_l), a component a row
    float4 xa[kPdMaxLinks];                   // x - a
    float qd_star[kPdMaxJoints], qd[kPdMaxJoints], qj[kPdMaxJoints];
    float padf[3 * IH_MAX_PADS];              // force sums over the frame's substeps
    float slip[8 * IH_MAX_PADS];              // per pad: w, w vt (3), w n (3), w spin
    unsigned short lbeg[32], lend[32];        // contact range of each link
};
static_assert(sizeof(PdSm) % 16 == 0, "the records that follow keep 16-byte alignment");

// Contact records by the contact's index, in arrays of `cap` entries rounded up to
// whole pairs of slots, so that a lane stores its slots' impulses without a test,
// and one more.
struct PdRecs {
    float4 *r, *n, *k, *lam, *mom;   // (r, gap), (n, link | pad << 8), (b, 1/k_n, 1/k_t, 0), lambda, (x + r) x lambda
    float4 *sph, *clc;               // sphere centres (clusters padded), cluster centres: world-rotated, relative to x; radius
    unsigned short *clp, *clist;     // surviving (link << 8 | cluster) pairs, contacts (link << 8 | sphere)
    int none;                        // an entry past the contacts, zero in lam and mom
};
__host__ __device__ constexpr int pd_round(int c_max) { return (c_max + 63) & ~63; }
__host__ __device__ constexpr int pd_clusters(int s_max) { return (s_max + kCluster - 1) / kCluster; }

__device__ __forceinline__ PdRecs pd_records(unsigned char *base, int s_max, int c_max) {
    const int cr = pd_round(c_max), ncl = pd_clusters(s_max);
    PdRecs q;
    q.none = cr;
    q.r = reinterpret_cast<float4 *>(base);
    q.n = q.r + cr;
    q.k = q.n + cr;
    q.lam = q.k + cr;
    q.mom = q.lam + cr + 1;
    q.sph = q.mom + cr + 1;
    q.clc = q.sph + ncl * kSphStride;
    q.clist = reinterpret_cast<unsigned short *>(q.clc + ncl);
    q.clp = q.clist + cr;
    return q;
}

// The fingers' kinematics at the joint angles S.qj, a lane per joint (lane 4 f + j:
// joint j of finger f, link 1 + 4 f + j): the sines of the finger's angles by its four
// lanes, then each lane runs the chain of finger_fk (hand.cuh) and keeps its own link and
// joint: joint 0 turns about +z through the root, joint j >= 1 by -q_j about link j's y
// axis through a_j, so its axis (for positive q_j) is -Q_j e_y.
__device__ __noinline__ void pd_fk(const DevScene &sc, PdSm &S, int lane) {
    const int f = lane >> 2, j = lane & 3;
    const bool on = f < sc.n_fingers;
    const float4 root = on ? sc.finger_root[f] : make_float4(0, 0, 0, 0);
    const float qa = on ? S.qj[lane] : 0.0f;
    float sn, cs;
    sincosf(j == 0 ? 0.5f * (root.w + qa) : -0.5f * qa, &sn, &cs);
    const float hs = 0.70710678118654752f;   // sin(pi/4) = cos(pi/4)
    const float s0 = __shfl_sync(kWarp, sn, lane & ~3), c0 = __shfl_sync(kWarp, cs, lane & ~3);
    Q4 Q = qmul({c0, 0.0f, 0.0f, s0}, {hs, 0.0f, -hs, 0.0f}), Qj = Q;
    V3 a = mk(root.x, root.y, root.z), aj = a;
#pragma unroll 1
    for (int i = 1; i < 4; ++i) {
        a = a + qrot(Q, mk(sc.link_len, 0, 0));
        const float si = __shfl_sync(kWarp, sn, (lane & ~3) + i), ci = __shfl_sync(kWarp, cs, (lane & ~3) + i);
        Q = qnorm(qmul(Q, {ci, 0.0f, si, 0.0f}));
        if (i == j) { Qj = Q; aj = a; }
    }
    if (on) {
        const V3 ax = qrot(Qj, mk(1, 0, 0));
        const V3 z = j == 0 ? mk(0, 0, 1) : qrot(Qj, mk(0, -1, 0));
        S.link[lane + 1][0] = make_float4(aj.x, aj.y, aj.z, 0.0f);
        S.link[lane + 1][1] = make_float4(ax.x, ax.y, ax.z, 0.0f);
        S.link[lane + 1][2] = make_float4(Qj.w, Qj.x, Qj.y, Qj.z);
        S.zax[lane] = make_float4(z.x, z.y, z.z, 0.0f);
        S.org[lane] = make_float4(aj.x, aj.y, aj.z, 0.0f);
    }
    if (lane == 31) {   // palm: identity pose at the origin
        S.link[0][0] = make_float4(0, 0, 0, 0);
        S.link[0][1] = make_float4(1, 0, 0, 0);
        S.link[0][2] = make_float4(1, 0, 0, 0);
    }
}

// The sum of v over the finger's joints from this lane's down to its first (lanes
// 4 f .. 4 f + 3 hold the finger's joints)
__device__ __forceinline__ V3 pd_prefix(V3 v, int lane) {
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
        const V3 o = mk(__shfl_up_sync(kWarp, v.x, off), __shfl_up_sync(kWarp, v.y, off), __shfl_up_sync(kWarp, v.z, off));
        const bool add = (lane & 3) >= off;
        v = {add ? v.x + o.x : v.x, add ? v.y + o.y : v.y, add ? v.z + o.z : v.z};
    }
    return v;
}
// ... and from this lane's up to its last
__device__ __forceinline__ V3 pd_suffix(V3 v, int lane) {
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
        const V3 o = mk(__shfl_down_sync(kWarp, v.x, off), __shfl_down_sync(kWarp, v.y, off), __shfl_down_sync(kWarp, v.z, off));
        const bool add = (lane & 3) + off < 4;
        v = {add ? v.x + o.x : v.x, add ? v.y + o.y : v.y, add ? v.z + o.z : v.z};
    }
    return v;
}

// The joints' lanes. SPLIT (at most 16 joints): lanes a and a + 16 hold joint a, the
// first its link's forces and angular velocity, the second the moments and linear
// velocity. Otherwise lane a holds all of joint a. z: the axis z_a, zo = z_a x o_a.
template <bool SPLIT>
struct PdJoint {
    V3 z, zo;
    float qs;          // qd*_a
    int a, beg, end;   // the joint, its link's contacts
    bool on, hi, more;
    const float4 *head[SPLIT ? kPdHead : 1];   // its first contacts' records (past the last: zeros)
    __device__ __forceinline__ void init(const PdSm &S, const PdRecs &q, int lane, int D) {
        a = SPLIT ? (lane & 15) : lane;
        hi = SPLIT && lane >= 16;
        on = a < D;
        z = zo = mk(0, 0, 0);
        qs = 0.0f;
        beg = end = 0;
        if (on) {
            z = xyz(S.zax[a]);
            zo = cross(z, xyz(S.org[a]));
            qs = S.qd_star[a];
            beg = S.lbeg[a + 1];
            end = S.lend[a + 1];
        }
        if (SPLIT) {
            const float4 *src = hi ? q.mom : q.lam;
#pragma unroll
            for (int k = 0; k < kPdHead; ++k) head[k] = src + (beg + k < end ? beg + k : q.none);
        }
        more = __any_sync(kWarp, end - beg > kPdHead);
    }
    // Every link's twist from the joint velocities: joint a adds (qd z_a, -qd z_a x o_a)
    // to the twist of every link it moves, so the twist of link a + 1 is the prefix over
    // the finger's joints up to a.
    __device__ __forceinline__ void twists(PdSm &S, int lane, float qd) const {
        if (SPLIT) {
            const V3 t = pd_prefix((hi ? zo : z) * (hi ? -qd : qd), lane);
            float *dst = S.tw[hi ? 3 : 0] + a + 1;
            if (on) { dst[0] = t.x; dst[32] = t.y; dst[64] = t.z; }
        } else {
            const V3 w = pd_prefix(z * qd, lane), c = pd_prefix(zo * (-qd), lane);
            if (on) {
                float *dst = S.tw[0] + a + 1;
                dst[0] = w.x; dst[32] = w.y; dst[64] = w.z; dst[96] = c.x; dst[128] = c.y; dst[160] = c.z;
            }
        }
    }
    // the joint's velocity under its links' impulses
    __device__ __forceinline__ float velocity(const PdRecs &q, int lane, float inv_Mj) const {
        float g;
        if (SPLIT) {
            V3 s0 = mk(0, 0, 0), s1 = s0;   // the contacts at even and odd places
            float4 v[kPdHead];
#pragma unroll
            for (int k = 0; k < kPdHead; ++k) v[k] = *head[k];
#pragma unroll
            for (int k = 0; k < kPdHead; k += 2) {
                s0 = s0 + xyz(v[k]);
                s1 = s1 + xyz(v[k + 1]);
            }
            if (more) {   // (some link holds more)
                const float4 *src = hi ? q.mom : q.lam;
#pragma unroll 1
                for (int ci = beg + kPdHead; ci < end; ci += 2) {
                    s0 = s0 + xyz(src[ci]);
                    s1 = s1 + xyz(src[ci + 1 < end ? ci + 1 : q.none]);
                }
            }
            const V3 s = pd_suffix(s0 + s1, lane);
            const float d = dot(s, hi ? z : zo), o = __shfl_xor_sync(kWarp, d, 16);
            g = hi ? d - o : o - d;
        } else {
            V3 F = mk(0, 0, 0), T = F;
#pragma unroll 1
            for (int ci = beg; ci < end; ++ci) {
                F = F + xyz(q.lam[ci]);
                T = T + xyz(q.mom[ci]);
            }
            // z . (T - o x F) = z . T - F . (z x o)
            F = pd_suffix(F, lane);
            T = pd_suffix(T, lane);
            g = dot(z, T) - dot(F, zo);
        }
        return on ? __fmaf_rn(-g, inv_Mj, qs) : 0.0f;
    }
};

__device__ __forceinline__ void put(float &t, int, float v) { t = v; }
__device__ __forceinline__ void put(F2 &t, int h, float v) { (h ? t.y : t.x) = v; }
__device__ __forceinline__ void put(Vec<float> &t, int, V3 v) { t = {v.x, v.y, v.z}; }
__device__ __forceinline__ void put(Vec<F2> &t, int h, V3 v) { put(t.x, h, v.x); put(t.y, h, v.y); put(t.z, h, v.z); }
__device__ __forceinline__ float4 get(const Vec<float> &t, int) { return make_float4(t.x, t.y, t.z, 0.0f); }
__device__ __forceinline__ float4 get(const Vec<F2> &t, int h) {
    return h ? make_float4(t.x.y, t.y.y, t.z.y, 0.0f) : make_float4(t.x.x, t.y.x, t.z.x, 0.0f);
}
__device__ __forceinline__ void add6(float (&acc)[6], const float (&s)[6]) {
#pragma unroll
    for (int q = 0; q < 6; ++q) acc[q] += s[q];
}
__device__ __forceinline__ void add6(float (&acc)[6], const F2 (&s)[6]) {
#pragma unroll
    for (int q = 0; q < 6; ++q) acc[q] = (acc[q] + s[q].x) + s[q].y;
}

// One (T = float) or two (T = float2: slots k, k + 1) of a lane's contacts, kept in
// registers over the iterations; slot k holds contact lane + 32 k. An empty slot
// (the palm at rest, r = 0, bias and 1/k 0) keeps a zero impulse and adds zeros.
// The bias velocity b n of slots 0 to 2 is rounded before it is subtracted, that of
// the contacts past them is not (a fused multiply-add): LAST tells that the unit
// holds some of those. A difference of rounding alone, kept for the results' bits (see
// prod_add), as is the order of tr K's two products.
template <typename T, bool LAST>
struct PdUnit {
    static constexpr int N = sizeof(T) / sizeof(float);
    Contact<T> c;
    Vec<T> p, nb;    // x + r; the bias velocity is -nb k
    Vec<T> w, v;     // the link's twist
    T k;
    int link[N], slot;
    __device__ __forceinline__ void load(const PdRecs &q, int slot_, int lane, int nc, V3 x) {
        slot = slot_;
        c.clear();
#pragma unroll
        for (int h = 0; h < N; ++h) {
            const int ci = lane + 32 * (slot + h);
            link[h] = 0;
            V3 r = mk(0, 0, 0), b = r;
            float kb = 1.0f;
            if (ci < nc) {
                const float4 n4 = q.n[ci], d = q.k[ci];
                const V3 n = xyz(n4);
                r = xyz(q.r[ci]);
                put(c.r, h, r);
                put(c.n, h, n);
                put(c.ikn, h, d.y);
                put(c.ikt, h, d.z);
                link[h] = __float_as_int(n4.w) & 0xff;
                if (LAST && slot + h >= 3) {
                    b = n * -1.0f;
                    kb = d.x;
                } else {
                    b = {-__fmul_rn(n.x, d.x), -__fmul_rn(n.y, d.x), -__fmul_rn(n.z, d.x)};
                }
            }
            put(p, h, x + r);
            put(nb, h, b);
            put(k, h, kb);
        }
    }
    // the links' twists, the update, and the impulses and moments to shared memory: in
    // turn for all of a lane's units, so that no load waits for another unit's stores
    __device__ __forceinline__ void gather(const PdSm &S) {
#pragma unroll
        for (int h = 0; h < N; ++h) {
            const float *t = &S.tw[0][link[h]];
            put(w, h, mk(t[0], t[32], t[64]));
            put(v, h, mk(t[96], t[128], t[160]));
        }
    }
    __device__ __forceinline__ void update(V3 vv, V3 ww, float mu_s, float inv_nc, float (&acc)[6]) {
        // the contact's target velocity: its link's at p less the bias along n
        const Vec<T> l = {t_add(t_fma(w.y, p.z, t_mul(t_neg(w.z), p.y)), v.x), t_add(t_fma(w.z, p.x, t_mul(t_neg(w.x), p.z)), v.y),
                          t_add(t_fma(w.x, p.y, t_mul(t_neg(w.y), p.x)), v.z)};
        if (LAST) c.c = {t_fma(nb.x, k, l.x), t_fma(nb.y, k, l.y), t_fma(nb.z, k, l.z)};
        else c.c = {t_add(l.x, nb.x), t_add(l.y, nb.y), t_add(l.z, nb.z)};
        c.update(vv, ww, mu_s, inv_nc);
        T s[6];
        c.wrench(s);
        add6(acc, s);
    }
    __device__ __forceinline__ void store(const PdRecs &q, int lane) const {
        const Vec<T> m = {t_fma(p.y, c.lam.z, t_mul(t_neg(p.z), c.lam.y)), t_fma(p.z, c.lam.x, t_mul(t_neg(p.x), c.lam.z)),
                          t_fma(p.x, c.lam.y, t_mul(t_neg(p.y), c.lam.x))};
#pragma unroll
        for (int h = 0; h < N; ++h) {   // (room to the end of the slot)
            q.lam[lane + 32 * (slot + h)] = get(c.lam, h);
            q.mom[lane + 32 * (slot + h)] = get(m, h);
        }
    }
};
struct PdNone {
    __device__ __forceinline__ void load(const PdRecs &, int, int, int, V3) {}
    __device__ __forceinline__ void gather(const PdSm &) {}
    __device__ __forceinline__ void update(V3, V3, float, float, float (&)[6]) {}
    __device__ __forceinline__ void store(const PdRecs &, int) const {}
};

// The iterations: the object's velocity enters as the prediction and leaves as the
// solution, the joints' as S.qd and the links' twists.
template <bool SPLIT>
struct PdSolve {
    PdSm &S;
    const PdRecs &q;
    const PdJoint<SPLIT> &jt;
    const S6 &Wi;
    V3 x, v_pred, w_pred;
    float inv_m, inv_Mj, mu_s, inv_nc;
    int lane, nc, iters;
    template <typename U0, typename U1, bool FURTHER>
    __device__ __forceinline__ void run(V3 &vv, V3 &ww) const {
        U0 u0;
        U1 u1;
        u0.load(q, 0, lane, nc, x);
        u1.load(q, 2, lane, nc, x);
        float qd = jt.qs;
#pragma unroll 1
        for (int it = 0; it < iters; ++it) {
            float acc[6] = {0, 0, 0, 0, 0, 0};
            u0.gather(S);
            u1.gather(S);
            u0.update(vv, ww, mu_s, inv_nc, acc);
            u1.update(vv, ww, mu_s, inv_nc, acc);
            u0.store(q, lane);
            u1.store(q, lane);
            if (FURTHER) {   // the contacts past the slots, in memory
#pragma unroll 1
                for (int ci = 32 * kPdSlots + lane; ci < nc; ci += 32) {
                    PdUnit<float, true> u;
                    u.load(q, ci >> 5, lane, nc, x);
                    const float4 l = q.lam[ci];
                    u.c.lam = {l.x, l.y, l.z};
                    u.gather(S);
                    u.update(vv, ww, mu_s, inv_nc, acc);
                    u.store(q, lane);
                }
            }
            __syncwarp();   // this iteration's impulses, for the joints' lanes
            qd = jt.velocity(q, lane, inv_Mj);
            width_sum6<32>(acc, kWarp, lane);
            vv = v_pred + mk(acc[0], acc[1], acc[2]) * inv_m;
            ww = w_pred + smul(Wi, mk(acc[3], acc[4], acc[5]));
            jt.twists(S, lane, qd);   // for the next iteration and the slip sensing
            __syncwarp();
        }
        if (jt.on && !jt.hi) S.qd[jt.a] = qd;
    }
};

template <bool SPLIT>
__global__ void __launch_bounds__(32, 8) pd_step_kernel(const __grid_constant__ PdArgs a, int s_max) {
    extern __shared__ __align__(16) unsigned char smem[];
    const DevScene &sc = a.sc;
    const DevConfig &cfg = a.cfg;
    const int lane = threadIdx.x;
    const int ns = cfg.substeps, Lk = sc.n_links, P = sc.n_pads, D = sc.n_joints;
    const float h = cfg.h, inv_h = 1.0f / h, inv_L = 1.0f / sc.link_len;
    const V3 grav = mk(cfg.gx * h, cfg.gy * h, cfg.gz * h);
    const float Mj = cfg.armature + h * cfg.kd + h * h * cfg.kp, inv_Mj = 1.0f / Mj;
    const int cap = cfg.c_max;
    const float inv_ns = 1.0f / (float)ns;
    // window mode (pose_frames != null): every frame's observation written out
    // for the frames' cost launches, the argmin taken afterwards
    const bool window_mode = a.pose_frames != nullptr;
    PdSm &S = *reinterpret_cast<PdSm *>(smem);
    const PdRecs q = pd_records(smem + sizeof(PdSm), s_max, cap);

    const int env = a.order ? __ldg(a.order + blockIdx.x) : (int)blockIdx.x;
    S.pads.build(sc, lane, 32);
    if (lane == 0) q.lam[q.none] = q.mom[q.none] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    int st = a.status[env];
    const float4 P0 = a.pose[2 * env], P1 = a.pose[2 * env + 1];
    const float4 V0 = a.vel[2 * env], V1 = a.vel[2 * env + 1];
    const float2 th = a.params[env];
    const int shp = a.shape[env];
    const int iters = a.iters[env];
    V3 x = xyz(P0);
    Q4 qt = {P1.x, P1.y, P1.z, P1.w};
    V3 v = xyz(V0), w = xyz(V1);
    const float m = th.x, mu = th.y, inv_m = 1.0f / m;
    const int sfirst = __ldg(sc.shape_first + shp), NS = __ldg(sc.shape_count + shp);
    const int ncl = (NS + kCluster - 1) / kCluster;
    const float inv_ncl = 1.0f / (float)ncl;
    const int cfirst = __ldg(sc.cl_first + shp);
    if (lane < D) {
        S.qj[lane] = a.qj[(size_t)env * D + lane];
        S.qd[lane] = a.qdj[(size_t)env * D + lane];
    }
    __syncwarp();

    unsigned long long work[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll 1
    for (int fr = 0; fr < a.n_frames; ++fr) {
#pragma unroll 1
        for (int k = lane; k < 3 * P; k += 32) S.padf[k] = 0.0f;
#pragma unroll 1
        for (int k = lane; k < 8 * P; k += 32) S.slip[k] = 0.0f;
        const int frame = a.frame0 + fr;
        const bool skip = (st & kDiverged) != 0;
#pragma unroll 1
        for (int s = 0; s < ns && !skip; ++s) {
            // -- 1. the hand at the substep start; the joints under the PD force alone
            pd_fk(sc, S, lane);
            const float frac = (float)(s + 1) / (float)ns;
            if (lane < D) {
                const float u0 = __ldg(a.cmd + (size_t)frame * D + lane), u1 = __ldg(a.cmd + (size_t)(frame + 1) * D + lane);
                const float u = u0 + frac * (u1 - u0);
                const float qs = (prod_add(cfg.armature, S.qd[lane], h * cfg.kp, u - S.qj[lane])) * inv_Mj;
                S.qd_star[lane] = qs;
                S.qd[lane] = qs;
            }
            const V3 v_pred = v + grav;
            const V3 w_pred = w;
            const M3 R = qmat(qt);
            S6 Jb;
            Jb.xx = __ldg(sc.shape_jinv + 6 * shp + 0); Jb.yy = __ldg(sc.shape_jinv + 6 * shp + 1);
            Jb.zz = __ldg(sc.shape_jinv + 6 * shp + 2); Jb.xy = __ldg(sc.shape_jinv + 6 * shp + 3);
            Jb.xz = __ldg(sc.shape_jinv + 6 * shp + 4); Jb.yz = __ldg(sc.shape_jinv + 6 * shp + 5);
            const S6 Wi = world_inv_inertia(R, Jb, inv_m);
#pragma unroll 1
            for (int j = lane; j < ncl * kCluster; j += 32) {
                float4 o = make_float4(kFar, kFar, kFar, 0.0f);   // (padding of the last cluster: far away)
                if (j < NS) {
                    const float4 s4 = __ldg(sc.spheres + sfirst + j);
                    const V3 cr = mmul(R, xyz(s4));
                    o = make_float4(cr.x, cr.y, cr.z, s4.w);
                }
                q.sph[(j >> 3) * kSphStride + (j & 7)] = o;
            }
#pragma unroll 1
            for (int k = lane; k < ncl; k += 32) {
                const float4 cl = __ldg(sc.clusters + cfirst + k);
                const V3 cr = mmul(R, xyz(cl));
                q.clc[k] = make_float4(cr.x, cr.y, cr.z, cl.w);
            }
            __syncwarp();
            if (lane < Lk) {
                const V3 xa = x - xyz(S.link[lane][0]);
                S.xa[lane] = make_float4(xa.x, xa.y, xa.z, 0.0f);
                S.lbeg[lane] = 0;
                S.lend[lane] = 0;
            }
            __syncwarp();

            // -- 2. cull (link, cluster) pairs by the clusters' enclosing spheres
            const int ncp = Lk * ncl;
            int nclp = 0;
#pragma unroll 1
            for (int p0 = 0; p0 < ncp; p0 += 32) {
                const int p = p0 + lane;
                bool keep = false;
                int e = 0;
                if (p < ncp) {
                    const int l = min((int)(((float)p + 0.5f) * inv_ncl), Lk - 1), k = p - l * ncl;
                    const float4 cc = q.clc[k];
                    keep = cluster_reaches(sc, cfg, l, xyz(S.xa[l]) + xyz(cc), cc.w, xyz(S.link[l][1]));
                    e = (l << 8) | k;
                }
                const unsigned bal = __ballot_sync(kWarp, keep);
                if (keep) q.clp[nclp + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)e;
                nclp += __popc(bal);
            }
            __syncwarp();
            // -- 2b. a lane tests the spheres of a surviving pair; the contacts in pair order
            int nc = 0;
#pragma unroll 1
            for (int e0 = 0; e0 < nclp; e0 += 32) {
                unsigned hits = 0;
                int e = 0;
                if (e0 + lane < nclp) {
                    e = q.clp[e0 + lane];
                    const int l = e >> 8, k = e & 0xff;
                    hits = cluster_hits(sc, cfg, l, k, xyz(S.xa[l]), xyz(S.link[l][1]), q.sph + k * kSphStride, NS, inv_L);
                }
                const int cnt = __popc(hits);
                int idx = nc;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const unsigned bal = __ballot_sync(kWarp, (cnt >> b) & 1);
                    idx += __popc(bal & ((1u << lane) - 1u)) << b;
                    nc += __popc(bal) << b;
                }
                const int cj = (e & 0xff00) | ((e & 0xff) * kCluster);
#pragma unroll
                for (int i = 0; i < kCluster; ++i) {
                    const int at = idx + __popc(hits & ((1u << i) - 1u));
                    if (((hits >> i) & 1u) && at < cap) q.clist[at] = (unsigned short)(cj + i);
                }
            }
            __syncwarp();
            if (nc > cap) {   // more contacts than the per-env capacity
                st |= IH_ENV_OVERFLOW;
                nc = 0;
            }
            work[0] += (unsigned)(nclp * kCluster);
            work[5] += (unsigned)ncp;
            work[1] += (unsigned)nc;
            work[2] += nc > 0 ? (unsigned long long)nc * iters : 0ull;
            work[3] += 1;
            work[4] += nc > 0 ? iters : 0;

            // -- 3. contact setup; each link's contact range (empty for links without contacts)
            const float trW = Wi.xx + Wi.yy + Wi.zz;
#pragma unroll 1
            for (int ci = lane; ci < nc; ci += 32) {
                const int e = q.clist[ci], l = e >> 8, j = e & 0xff;
                if (ci == 0 || q.clist[ci - 1] >> 8 != l) S.lbeg[l] = (unsigned short)ci;
                if (ci == nc - 1 || q.clist[ci + 1] >> 8 != l) S.lend[l] = (unsigned short)(ci + 1);
                const float4 s4 = q.sph[(j >> 3) * kSphStride + (j & 7)];
                const V3 cr = xyz(s4), ca = xyz(S.xa[l]) + cr;
                const float4 lq = S.link[l][2];
                const Hit hh = l == 0 ? hit_box_local(ca, s4.w, sc.palm_hx, sc.palm_hy, sc.palm_hz)
                                      : hit_capsule(ca, s4.w, xyz(S.link[l][1]), sc.link_len, inv_L, sc.link_rad,
                                                    {lq.x, lq.y, lq.z, lq.w});
                const V3 n = hh.n, r = cr - n * s4.w;
                const V3 rn = cross(r, n);
                float kn = inv_m + dot(rn, smul(Wi, rn));
                float trK = prod_add(dot(r, r), trW, 3.0f, inv_m) - dot(r, smul(Wi, r));
                const V3 p = x + r;
                const int f4 = (l - 1) & ~3;
#pragma unroll 1
                for (int ja = f4; ja < l; ++ja) {   // the joints that move the link (none of the palm)
                    if (l == 0) break;
                    const V3 J = cross(xyz(S.zax[ja]), p - xyz(S.org[ja]));
                    const float jn = dot(J, n);
                    kn = __fmaf_rn(jn * jn, inv_Mj, kn);
                    trK = __fmaf_rn(dot(J, J), inv_Mj, trK);
                }
                q.r[ci] = make_float4(r.x, r.y, r.z, hh.gap);
                q.n[ci] = make_float4(n.x, n.y, n.z, __int_as_float(l | (S.pads.find(l, hh.t) << 8)));
                q.k[ci] = make_float4(contact_bias(cfg, hh.gap), 1.0f / kn, 2.0f / (trK - kn), 0.0f);
                q.lam[ci] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
            __syncwarp();

            // -- 4. Jacobi iterations over the object and the joints
            V3 vv = v_pred, ww = w_pred;
            if (nc > 0) {
                // the links' twists under the PD prediction alone (palm: at rest)
                if (lane < 6) S.tw[lane][0] = 0.0f;
                PdJoint<SPLIT> jt;
                jt.init(S, q, lane, D);
                jt.twists(S, lane, jt.qs);
                __syncwarp();
                const PdSolve<SPLIT> solve = {S, q, jt, Wi, x, v_pred, w_pred, inv_m, inv_Mj, 4096.0f * mu, 1.0f / (float)nc,
                                              lane, nc, iters};
                // one loop per number of occupied slots, each a straight stretch of code
                if (nc <= 32) solve.template run<PdUnit<float, false>, PdNone, false>(vv, ww);
                else if (nc <= 64) solve.template run<PdUnit<F2, false>, PdNone, false>(vv, ww);
                else if (nc <= 96) solve.template run<PdUnit<F2, false>, PdUnit<float, false>, false>(vv, ww);
                else if (nc <= 32 * kPdSlots) solve.template run<PdUnit<F2, false>, PdUnit<F2, true>, false>(vv, ww);
                else solve.template run<PdUnit<F2, false>, PdUnit<F2, true>, true>(vv, ww);
                __syncwarp();
            }
            v = vv;
            w = ww;

            // -- 5. integrate the object and the joints (contact points stay
            //       those of the substep start: p = x_s + r)
            const V3 x_s = x;
            x = x + v * h;
            {
                const float wn = sqrtf(dot(w, w));
                float sn, cs;
                sincosf(0.5f * wn * h, &sn, &cs);
                const float kq = (wn > 0.0f) ? sn / wn : 0.5f * h;
                qt = qnorm(qmul({cs, w.x * kq, w.y * kq, w.z * kq}, qt));
            }
            // (S.tw holds the links' twists at the final joint velocities)
            if (lane < D) S.qj[lane] += h * S.qd[lane];
            // pads: force -lambda / h per contact, and the slip sums weighted
            // by the normal impulse
            if (lane < P) {
                const int p = lane, l = __ldg(sc.pad_link + p);
                float fx = 0.0f, fy = 0.0f, fz = 0.0f;
                float sw = 0.0f, s1x = 0.0f, s1y = 0.0f, s1z = 0.0f, snx = 0.0f, sny = 0.0f, snz = 0.0f, ssp = 0.0f;
                const float *t = &S.tw[0][l];
                const V3 wl = mk(t[0], t[32], t[64]), cl = mk(t[96], t[128], t[160]);
                const int e = S.lend[l];
#pragma unroll 1
                for (int ci = S.lbeg[l]; ci < e; ++ci) {
                    const float4 n4 = q.n[ci];
                    if (((__float_as_int(n4.w) >> 8) & 0xff) != p) continue;
                    const V3 lam = xyz(q.lam[ci]), r = xyz(q.r[ci]), n = xyz(n4);
                    fx -= lam.x * inv_h; fy -= lam.y * inv_h; fz -= lam.z * inv_h;
                    const float ln = dot(lam, n);
                    if (!(ln > 0.0f)) continue;
                    const V3 vrel = (v + cross(w, r)) - (cross(wl, x_s + r) + cl);
                    const V3 vt = vrel - n * dot(vrel, n);
                    const float spin = dot(w - wl, n);
                    sw += ln;
                    s1x += ln * vt.x; s1y += ln * vt.y; s1z += ln * vt.z;
                    snx += ln * n.x; sny += ln * n.y; snz += ln * n.z;
                    ssp += ln * spin;
                }
                S.padf[3 * p] += fx; S.padf[3 * p + 1] += fy; S.padf[3 * p + 2] += fz;
                float *A = S.slip + 8 * p;
                A[0] += sw; A[1] += s1x; A[2] += s1y; A[3] += s1z; A[4] += snx; A[5] += sny; A[6] += snz; A[7] += ssp;
            }
            __syncwarp();
        }
        if (!skip) {
            bool fin = all_finite(x, qt, v, w);
            if (lane < D) fin = fin && isfinite(S.qj[lane]) && isfinite(S.qd[lane]);
            fin = __all_sync(kWarp, fin);
            if (!fin) st |= IH_ENV_NONFINITE;
            else if (dot(x, x) > cfg.escape_radius * cfg.escape_radius) st |= IH_ENV_ESCAPED;
        }
        // the observation of the frame just stepped (pad poses from the joints
        // at its end, slip from the frame's sums), of every frame in window mode
        const bool last = fr == a.n_frames - 1;
        if (!window_mode && !last) continue;
        pd_fk(sc, S, lane);
        __syncwarp();
        const size_t ef = (size_t)fr * a.N + env;
        if (lane < P) {
            const int p = lane, l = __ldg(sc.pad_link + p);
            const float4 A0 = S.link[l][0], Aq = S.link[l][2];
            const Q4 lq = {Aq.x, Aq.y, Aq.z, Aq.w};
            V3 c;
            if (l == 0) {
                c = xyz(A0) + qrot(lq, mk(0, 0, sc.palm_hz));
            } else {
                const float s1 = fminf(__ldg(sc.pad_s1 + p), 1.0f), s0 = fmaxf(__ldg(sc.pad_s0 + p), 0.0f);
                c = xyz(A0) + qrot(lq, mk(0.5f * (s0 + s1) * sc.link_len, 0, 0));
            }
            const float *A = S.slip + 8 * p;
            float dx = 0.0f, dy = 0.0f;
            int flags = 0;
            if (A[0] > 0.0f) {
                const float iw = 1.0f / A[0];
                const V3 vt = mk(A[1], A[2], A[3]) * iw;
                V3 nb = mk(A[4], A[5], A[6]);
                nb = nb * rsqrtf(dot(nb, nb));
                const float spin = A[7] * iw;
                if (sqrtf(dot(vt, vt)) > cfg.v_slip) {
                    const V3 ax = xyz(S.link[l][1]);
                    V3 e1 = ax - nb * dot(ax, nb);
                    e1 = e1 * rsqrtf(dot(e1, e1));
                    const V3 e2 = cross(nb, e1);
                    const float d1 = dot(vt, e1), d2 = dot(vt, e2), idn = rsqrtf(d1 * d1 + d2 * d2);
                    dx = d1 * idn;
                    dy = d2 * idn;
                    flags |= 1;
                }
                if (fabsf(spin) > cfg.w_slip) flags |= (spin > 0.0f) ? 6 : 2;
            }
            const float4 pp = make_float4(c.x, c.y, c.z, 0.0f), sl = make_float4(dx, dy, __int_as_float(flags), 0.0f);
            if (window_mode) {
                a.fo_pp[2 * (ef * P + p)] = pp;
                a.fo_pp[2 * (ef * P + p) + 1] = Aq;
                a.fo_slip[ef * P + p] = sl;
            }
            if (last) {
                a.pad_pose[2 * ((size_t)env * P + p)] = pp;
                a.pad_pose[2 * ((size_t)env * P + p) + 1] = Aq;
                a.slip[(size_t)env * P + p] = sl;
            }
        }
#pragma unroll 1
        for (int k = lane; k < 3 * P; k += 32) {
            const float f = S.padf[k] * inv_ns;
            if (window_mode) a.fo_forces[ef * 3 * P + k] = f;
            if (last) a.forces[(size_t)env * P * 3 + k] = f;
        }
        if (window_mode) {
            if (lane < D) a.fo_q[ef * D + lane] = S.qj[lane];
            if (lane == 0) {
                a.fo_status[ef] = st;
                a.pose_frames[2 * ef] = make_float4(x.x, x.y, x.z, 0.0f);
                a.pose_frames[2 * ef + 1] = make_float4(qt.w, qt.x, qt.y, qt.z);
            }
        }
        __syncwarp();
    }
    if (lane < D) {
        a.qj[(size_t)env * D + lane] = S.qj[lane];
        a.qdj[(size_t)env * D + lane] = S.qd[lane];
    }
    if (lane == 0) {
        a.pose[2 * env] = make_float4(x.x, x.y, x.z, 0.0f);
        a.pose[2 * env + 1] = make_float4(qt.w, qt.x, qt.y, qt.z);
        a.vel[2 * env] = make_float4(v.x, v.y, v.z, 0.0f);
        a.vel[2 * env + 1] = make_float4(w.x, w.y, w.z, 0.0f);
        a.status[env] = st;
        if (a.work)
            for (int k = 0; k < 6; ++k)
                if (work[k]) atomicAdd(a.work + k, work[k]);
    }
}

// every environment's hand at rest at q0 (D values; null: zero)
__global__ void hand_rest_kernel(int N, int D, const float *q0, float *qj, float *qdj) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (size_t)N * D) return;
    qj[k] = q0 ? q0[k % D] : 0.0f;
    qdj[k] = 0.0f;
}

}  // namespace

cudaError_t launch_hand_rest(int N, int D, const float *q0, float *qj, float *qdj, cudaStream_t s) {
    const size_t n = (size_t)N * D;
    if (n == 0) return cudaSuccess;
    hand_rest_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(N, D, q0, qj, qdj);
    return cudaGetLastError();
}

size_t pd_step_smem_bytes(int s_max, int c_max) {
    const size_t cr = pd_round(c_max), ncl = pd_clusters(s_max);
    return sizeof(PdSm) + (5 * cr + 2 + ncl * (kSphStride + 1)) * sizeof(float4) +
           ((cr + kPdMaxLinks * ncl) * sizeof(unsigned short) + 15) / 16 * 16;
}

cudaError_t pd_step_prepare(int s_max, int c_max) {
    const size_t bytes = pd_step_smem_bytes(s_max, c_max);
    if (bytes <= 48 * 1024) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(pd_step_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(pd_step_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    return e;
}

// a block of one warp per environment
cudaError_t launch_pd_step(const PdArgs &a, int s_max, cudaStream_t s) {
    const size_t bytes = pd_step_smem_bytes(s_max, a.cfg.c_max);
    if (a.sc.n_joints <= 16) pd_step_kernel<true><<<a.N, 32, bytes, s>>>(a, s_max);
    else pd_step_kernel<false><<<a.N, 32, bytes, s>>>(a, s_max);
    return cudaGetLastError();
}

}  // namespace ih
