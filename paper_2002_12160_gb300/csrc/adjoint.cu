// adjoint.cu -- reverse-mode derivative of the tracking cost with respect to
// each environment's initial pose, mass and friction coefficient.
//
// The cost of one environment over the frames [frame0, frame0 + H) is
//     L = sum_f sum_l w_force |c_f^(l) - o_f^(l)|^2  (+ contact-state terms)
// -- the tracking cost of Sec. III-C on the simulated pad forces c_f of the
// frame step s_{t+1} = f(s_t, u_t, theta) of Sec. III-A. The contact-state
// terms are piecewise constant and carry no derivative. The gradient is taken
// by hand-written reverse mode through every operation of the step: sphere
// positions, narrowphase gaps, normals and lever arms, effective masses, bias
// and link velocities, the fixed number of projected Jacobi iterations, and
// the integrator (the same expressions as step_kernel.cuh, through contact.cuh; a few
// sums are rounded in another order, so the forwards agree up to rounding).
//
// The projections of the Jacobi update are not differentiable on the cone's
// boundary. The reverse sweep therefore uses smooth stand-ins for their
// derivatives only; the forward values stay exact:
//   * normal clamp max(0, z): the derivative sigmoid(beta z) of a softplus;
//   * radial clamp of the tangential impulse z onto the disk of radius L:
//     the derivative of z smin(|z|, L) / |z| with
//     smin(a, b) = (a + b - sqrt((a - b)^2 + (w b)^2)) / 2.
// Contact membership (gap < margin), the capsule's end clamps, the palm's face
// or clamp pattern and the bias regimes are held fixed.
//
// Work layout: a block of GW warps (32 GW threads; 4 or 1) per environment. The
// block enumerates the contacts together, in the step's order (a thread tests the
// eight spheres of a (link, cluster) pair that survived the cull); thread k % (32 GW)
// then owns contact k for the setup, the Jacobi iterations and their reverse --
// 128 contacts of a block in registers and shared memory, the further ones (with one
// warp) in the environment's scratch memory -- and the block sums impulses and derivatives
// by warp shuffles and a shared-memory exchange between its warps. The state
// at every K-th frame is kept (checkpoints). The reverse sweep walks the
// segments between checkpoints backwards: it recomputes the segment's
// substep start states and pad forces from its checkpoint while recording the
// tape (the impulses after every Jacobi iteration and the per-iteration
// impulse sums) of every substep of the segment, then runs the substeps'
// reverse sweeps in reverse order. When the whole segment's tape does not fit
// the handle's budget, each substep is run once more just before its reverse
// sweep to record its tape alone; the results are the same bit for bit. (The
// last segment's tape is recorded by the first pass itself.) Checkpoints,
// segment states and the tape live in a slice of a scratch buffer owned by
// the handle, one slice per environment.
//
// What bounds it: an iteration and its reverse are one chain of dependent
// arithmetic and shuffles per environment (two or fewer warps a scheduler at 255
// registers), and where many environments run, also the instruction fetch, since
// every warp is somewhere else in the code. Hence: two contacts of a lane packed
// in FP32 pairs (half the instructions); one loop per number of occupied slots,
// each body one straight stretch of code (predicated stores and copies instead of
// branches), so that the scheduler overlaps the chains: an iteration of the reverse
// 1100 -> 650 cycles for four warps with a contact a thread; the tape read by
// asynchronous copies three iterations ahead; everything off those loops rolled.
// Against one thread per pair, scalar slots with a branch each, and tape loads in the
// iteration that needs them, at the public call: 1024 cylinders, 30 frames, three
// segments 5.28 -> 4.28 ms; 102 cylinders, 10 frames, 552 -> 455 us; 64 boxes, 5 frames
// (bound by the host), the kernel 258 -> 200 us.
#include <type_traits>

#include "contact.cuh"
#include "internal.cuh"

namespace ih {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRC = 128;   // contacts of a block held in registers and shared memory (a thread's first, with four warps)
// The compiled shapes GW: one warp (1), four warps for scenes of at most kRC contacts
// (4), and four warps whose threads hold a second contact (kTwo), so that no contact of
// theirs is in memory
constexpr int kTwo = 4 | 8;
template <int GW>
constexpr int kWarps = GW & 7;
template <int GW>
constexpr int kHeld = GW == kTwo ? 2 * kRC : kRC;
static_assert(IH_MAX_CONTACTS <= kHeld<kTwo>, "two contacts a thread hold all");
// Iterations of the tape held in shared memory by the reverse sweep, copied there
// asynchronously three iterations ahead. (Requested into registers an iteration
// ahead, the rotation of the registers waited for the loads: 990 cycles an
// iteration for four warps with a contact a thread.)
constexpr int kRing = 4;
// (bytes: 16, or 0 to fill with zeros; skipped without a branch unless `on`)
__device__ __forceinline__ void copy_async(float4 *dst, const float4 *src, int bytes, bool on = true) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.s32 p, %3, 0;\n@p cp.async.ca.shared.global [%0], [%1], 16, %2;\n}" ::"r"(
            (unsigned)__cvta_generic_to_shared(dst)),
        "l"(src), "r"(bytes), "r"((int)on)
        : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// a store without a branch (`on` varies by lane), so that a loop's body stays one
// stretch of code for the scheduler
__device__ __forceinline__ void store_if(bool on, float4 *dst, float4 v) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.s32 p, %5, 0;\n@p st.global.v4.f32 [%0], {%1, %2, %3, %4};\n}" ::"l"(dst), "f"(v.x),
                 "f"(v.y), "f"(v.z), "f"(v.w), "r"((int)on)
                 : "memory");
}
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The warps of one environment (a block): thread gt, lane, warp; sync() is the
// block's barrier.
template <int GW>
struct AGroup {
    static constexpr int T = 32 * kWarps<GW>;
    int gt, lane, wg;
    __device__ AGroup() {
        gt = threadIdx.x;
        lane = threadIdx.x & 31;
        wg = gt >> 5;
    }
    __device__ __forceinline__ void sync() const {
        if constexpr (GW == 1) __syncwarp();
        else __syncthreads();
    }
};

template <bool V>
struct Flag {
    static constexpr bool value = V;
};

struct Body {
    V3 x;
    Q4 q;
    V3 v, w;
};
struct Adj {   // derivatives of the cost w.r.t. a Body's components
    V3 x;
    Q4 q;
    V3 v, w;
};

__device__ __forceinline__ void store_body(float4 *p, const Body &b) {
    p[0] = make_float4(b.x.x, b.x.y, b.x.z, 0.0f);
    p[1] = make_float4(b.q.w, b.q.x, b.q.y, b.q.z);
    p[2] = make_float4(b.v.x, b.v.y, b.v.z, 0.0f);
    p[3] = make_float4(b.w.x, b.w.y, b.w.z, 0.0f);
}
__device__ __forceinline__ Body load_body(const float4 *p) {
    const float4 a = p[0], b = p[1], c = p[2], d = p[3];
    return Body{xyz(a), Q4{b.x, b.y, b.z, b.w}, xyz(c), xyz(d)};
}
__device__ __forceinline__ Q4 qconj(Q4 q) { return {q.w, -q.x, -q.y, -q.z}; }

// The forward substep's quaternion product and world inverse inertia, whose
// contraction differs from the step's (internal.cuh) in the places named: by rounding
// alone, kept for the gradients' and costs' bits (see prod_add)
__device__ __forceinline__ Q4 qmul_f(Q4 a, Q4 b) {
    return {__fmaf_rn(-a.z, b.z, __fmaf_rn(-a.y, b.y, prod_sub(a.w, b.w, a.x, b.x))),
            __fmaf_rn(-a.z, b.y, __fmaf_rn(a.y, b.z, prod_add(a.x, b.w, a.w, b.x))),    // (a.w b.x rounded first)
            __fmaf_rn(a.z, b.x, __fmaf_rn(a.y, b.w, prod_sub(a.w, b.y, a.x, b.z))),
            __fmaf_rn(a.z, b.w, __fmaf_rn(-a.y, b.x, prod_add(a.x, b.y, a.w, b.z)))};   // (a.w b.z)
}
__device__ __forceinline__ S6 world_inv_inertia_f(const M3 &R, const S6 &J, float inv_m) {
    const V3 r0 = {R.c0.x, R.c1.x, R.c2.x}, r1 = {R.c0.y, R.c1.y, R.c2.y}, r2 = {R.c0.z, R.c1.z, R.c2.z};
    const V3 a0 = {__fmaf_rn(J.xz, r0.z, prod_add(J.xy, r0.y, J.xx, r0.x)), __fmaf_rn(J.yz, r0.z, prod_add(J.yy, r0.y, J.xy, r0.x)),
                   __fmaf_rn(J.zz, r0.z, prod_add(J.xz, r0.x, J.yz, r0.y))};   // (first and second row)
    return sandwich(r0, r1, r2, a0, smul(J, r1), smul(J, r2), inv_m);
}
struct Centres {
    float4 sph[IH_MAX_SPHERES / kCluster * kSphStride];   // the substep's sphere centres (world rotation, relative to x), radius
    float4 clc[IH_MAX_SPHERES / kCluster];   // cluster centres (likewise), enclosing radius
    unsigned short clp[kMaxLinks * (IH_MAX_SPHERES / kCluster)];   // surviving (link << 8 | cluster) pairs
};
template <int GW>
struct alignas(16) GroupSm {
    // GW = 1: the constants of the lane's contacts lane + 32 k (k < 4), slots 2 p
    // and 2 p + 1 interleaved so that a float4 holds two pairs: r, n, c, 1/k_n, 1/k_t
    float4 cp[GW == 1 ? 2 : 1][6][32];
    float4 clam[kRC];              // the pass's final impulses (pad sums)
    float4 meta[kRC];              // reverse: the contacts' gap, link | pad << 8 and sphere
    union {                        // (a substep's enumeration and a reverse sweep never overlap)
        float4 ring[kRing][kHeld<GW>];   // reverse: the impulses after iterations it & (kRing - 1), on their way from the tape
        Centres en;                // forward: the enumeration's centres and pairs
    };
    float4 rsum[kWarps<GW>][kRing][2];     // ... and their sums, a copy per warp
    float4 xa[kMaxLinks], ax[kMaxLinks];     // x - link origin, link axis
    double term[IH_MAX_PADS];      // a frame's FP64 force term of each pad
    float padacc[IH_MAX_PADS * 3];
    float fbar[IH_MAX_PADS * 3];   // dL/dF_p / (h ns): minus the derivative w.r.t. a final impulse
    float4 red[2][kWarps<GW>][2];          // partial sums of the block's warps (double-buffered)
    float fin[16];                 // results of the contacts' warps for the others
    int cnt[2][kWarps<GW>];                // hits of each warp in a compaction round (double-buffered)
    int flag[IH_MAX_PADS];         // a frame's contact-state mismatch of each pad
    unsigned short lbeg[kMaxLinks], lend[kMaxLinks];   // contact range of each link
    unsigned short clist[IH_MAX_CONTACTS];   // the contacts in order (link << 8 | sphere)
    unsigned char cpad[IH_MAX_CONTACTS];     // their pads
};

// Sum of `mine` (0..15) over the block's threads before this one (returned, plus
// base) and over all of them (added to base): the slots of an order-preserving
// compaction, by bit planes of the warps' ballots.
template <int GW, int BITS>
__device__ __forceinline__ int gcompact(int mine, int &base, const AGroup<GW> &G, GroupSm<GW> &S, int &parity) {
    int off = base, tot = 0;
#pragma unroll
    for (int b = 0; b < BITS; ++b) {
        const unsigned bal = __ballot_sync(kFull, (mine >> b) & 1);
        off += __popc(bal & ((1u << G.lane) - 1u)) << b;
        tot += __popc(bal) << b;
    }
    if constexpr (GW > 1) {
        int *c = S.cnt[parity];
        if (G.lane == 0) c[G.wg] = tot;
        G.sync();
        tot = 0;
#pragma unroll
        for (int w = 0; w < kWarps<GW>; ++w) {
            const int k = c[w];
            if (w < G.wg) off += k;
            tot += k;
        }
        parity ^= 1;
    }
    base += tot;
    return off;
}

// Sum of 6 values over the first aw warps of the block, every one of their threads
// receiving the sums: within each warp by shuffles, then the warps' partials in
// warp order.
template <int GW>
__device__ __forceinline__ void gsum6(float (&v)[6], const AGroup<GW> &G, GroupSm<GW> &S, int &parity, int aw = kWarps<GW>) {
    if constexpr (GW == 1) {
        width_sum6<32>(v, kFull, G.lane);
    } else {
        const float c = width_scatter6<32>(v, kFull, G.lane);
        float *r = reinterpret_cast<float *>(&S.red[parity][0][0]);
        const int k = G.lane >> 2;
        if ((G.lane & 3) == 0 && k < 6) r[G.wg * 8 + k] = c;
        asm volatile("bar.sync 1, %0;" ::"r"(32 * aw) : "memory");
        const float4 *r4 = reinterpret_cast<const float4 *>(r);
        float4 lo = r4[0], hi = r4[1];
#pragma unroll
        for (int w = 1; w < kWarps<GW>; ++w) {
            const float4 l = r4[2 * w], u = r4[2 * w + 1];
            const bool on = w < aw;   // (the others' places hold old sums)
            lo.x += on ? l.x : 0.0f; lo.y += on ? l.y : 0.0f; lo.z += on ? l.z : 0.0f; lo.w += on ? l.w : 0.0f;
            hi.x += on ? u.x : 0.0f; hi.y += on ? u.y : 0.0f;
        }
        v[0] = lo.x; v[1] = lo.y; v[2] = lo.z; v[3] = lo.w; v[4] = hi.x; v[5] = hi.y;
        parity ^= 1;
    }
}

// Per-slot scratch layout in floats (every part starts on a float4 boundary):
// checkpoints, a segment's substep start states, every frame's pad forces, the
// impulses of a pass (final ones for the pad sums; the running ones of the
// contacts past the register slots), the reverse state of the contacts past
// the register slots, the contact count of every taped substep, the contact
// records and counts of the nrec substeps of the segments that are
// recomputed (their recomputation replays them), then nblk tape blocks of
// (contact records, impulse after each iteration, iteration sums): one block
// per substep of a segment when the whole segment is taped, else a single
// block re-filled substep by substep.
struct SlotLayout {
    size_t ck, sg, sf, lamf, adj, ncs, recs, nrc, tape, blk_rec, blk_lamh, blk_sh, blk_stride, total;
};
__host__ __device__ inline size_t round4(size_t x) { return (x + 3) & ~size_t(3); }
__host__ __device__ inline SlotLayout slot_layout(int H, int K, int ns, int P, int cap, int iters_max, int nblk,
                                                  int nrec) {
    SlotLayout L;
    size_t o = 0;
    const size_t nck = (size_t)((H + K - 1) / K);
    L.ck = o;   o += round4(nck * 16);                        // checkpoint states
    L.sg = o;   o += round4((size_t)K * ns * 16);             // substep start states of a segment
    L.sf = o;   o += round4((size_t)H * P * 3);               // pad forces of every frame
    L.lamf = o; o += round4((size_t)cap * 4);                 // impulses of a pass
    L.adj = o;  o += round4((size_t)cap * 16);                // reverse state of the contacts in memory
    L.ncs = o;  o += round4((size_t)K * ns);                  // contacts of each taped substep (int)
    L.recs = o; o += (size_t)nrec * cap * 16;                 // records of the recomputed segments' substeps
    L.nrc = o;  o += round4((size_t)nrec);                    // their contact counts (int)
    L.blk_rec = 0;
    L.blk_lamh = round4((size_t)cap * 16);                                   // contact records
    L.blk_sh = L.blk_lamh + round4((size_t)iters_max * cap * 4);             // impulse after each iteration
    L.blk_stride = L.blk_sh + round4((size_t)(iters_max > 0 ? iters_max : 1) * 8);   // sums after each iteration
    L.tape = o; o += (size_t)nblk * L.blk_stride;
    L.total = o;
    return L;
}

struct SlotPtr {
    float4 *ck, *sg, *rec, *lamh, *lamf;
    float4 *recs;   // records of substep q of the recomputed segments at recs + q * cap * 4
    int *nrc;       // their contact counts
    float4 *adjs;   // per contact past the register slots: (lb, 1/k_n bar), (nb, 1/k_t bar), (rb, -), (cb, -)
    float *sf, *sh;
    int *ncs;
    float *tape;
    size_t blk_lamh, blk_sh, blk_stride;
    // the same slot with its tape pointers on block b
    __device__ SlotPtr blk(int b) const {
        SlotPtr q = *this;
        float *t = tape + (size_t)b * blk_stride;
        q.rec = reinterpret_cast<float4 *>(t);
        q.lamh = reinterpret_cast<float4 *>(t + blk_lamh);
        q.sh = t + blk_sh;
        return q;
    }
};

// Per-environment constants.
struct Env {
    int sfirst, NS, iters, cfirst;
    float mu, inv_m;
    S6 Jb;
};

// contact record: [0] (r, gap) [1] (n, 1/k_n) [2] (c, 1/k_t) [3] (t, link | pad << 8, sphere, -)
__device__ __forceinline__ int rec_pad(float4 r3) { return (__float_as_int(r3.y) >> 8) & 0xff; }   // (of GroupSm::meta too)

// A pair's constants in shared memory (GroupSm::cp): value v of r, n, c, 1/k_n,
// 1/k_t (0..10) of slots 2 p and 2 p + 1
template <int GW>
__device__ __forceinline__ void cp_store(GroupSm<GW> &S, int slot, int lane, V3 r, V3 n, V3 c, float ikn, float ikt) {
    const float v[11] = {r.x, r.y, r.z, n.x, n.y, n.z, c.x, c.y, c.z, ikn, ikt};
#pragma unroll
    for (int q = 0; q < 11; ++q)
        reinterpret_cast<float *>(&S.cp[GW == 1 ? slot >> 1 : 0][q >> 1][lane])[(q & 1) * 2 + (slot & 1)] = v[q];
}
template <int GW>
__device__ __forceinline__ void cp_load(const GroupSm<GW> &S, int slot, int lane, Contact<F2> &c) {
    const float4 *p = &S.cp[GW == 1 ? slot >> 1 : 0][0][lane];
    const float4 a = p[0], b = p[32], d = p[64], e = p[96], f = p[128], g = p[160];
    c.r = {{a.x, a.y}, {a.z, a.w}, {b.x, b.y}};
    c.n = {{b.z, b.w}, {d.x, d.y}, {d.z, d.w}};
    c.c = {{e.x, e.y}, {e.z, e.w}, {f.x, f.y}};
    c.ikn = {f.z, f.w};
    c.ikt = {g.x, g.y};
}
template <int GW>
__device__ __forceinline__ void cp_load(const GroupSm<GW> &S, int slot, int lane, Contact<float> &c) {   // slot even
    Contact<F2> t;
    cp_load(S, slot, lane, t);
    c.r = {t.r.x.x, t.r.y.x, t.r.z.x};
    c.n = {t.n.x.x, t.n.y.x, t.n.z.x};
    c.c = {t.c.x.x, t.c.y.x, t.c.z.x};
    c.ikn = t.ikn.x;
    c.ikt = t.ikt.x;
}
// The constants of a thread's second contact (four warps; empty: adds zeros)
template <int GW>
__device__ __forceinline__ void load_second(const SlotPtr &sp, const AGroup<GW> &G, int nc, Contact<float> &own2) {
    own2.clear();
    const int ci = kRC + G.gt;
    if (ci < nc) {
        const float4 r0 = sp.rec[4 * ci], r1 = sp.rec[4 * ci + 1], r2 = sp.rec[4 * ci + 2];
        own2.r = {r0.x, r0.y, r0.z};
        own2.n = {r1.x, r1.y, r1.z};
        own2.c = {r2.x, r2.y, r2.z};
        own2.ikn = r1.w;
        own2.ikt = r2.w;
    }
}
// The constants of the block's first kRC contacts from their records: to shared
// memory (GW = 1, every load requested before the first is used; empty slots to
// the next whole pair), or to the thread's own contact; with META the rest of the
// record too
template <int GW, bool META>
__device__ __forceinline__ void load_constants(const SlotPtr &sp, GroupSm<GW> &S, const AGroup<GW> &G, int nc, Contact<float> &own) {
    constexpr int NK = GW == 1 ? 4 : 1;
    float4 r[NK][4];
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        const int ci = G.gt + AGroup<GW>::T * k;
        r[k][0] = r[k][2] = r[k][3] = make_float4(0, 0, 0, 0);
        r[k][1] = make_float4(0, 0, 1, 0);
        if (ci < nc)
            for (int q = 0; q < (META ? 4 : 3); ++q) r[k][q] = sp.rec[4 * ci + q];
    }
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        const int ci = G.gt + AGroup<GW>::T * k;
        if (META && ci < nc) S.meta[ci] = make_float4(r[k][0].w, r[k][3].y, r[k][3].z, 0.0f);
        if constexpr (GW == 1) {
            if (32 * (k & ~1) < nc) cp_store(S, k, G.lane, xyz(r[k][0]), xyz(r[k][1]), xyz(r[k][2]), r[k][1].w, r[k][2].w);
        } else {
            own.r = {r[k][0].x, r[k][0].y, r[k][0].z};
            own.n = {r[k][1].x, r[k][1].y, r[k][1].z};
            own.c = {r[k][2].x, r[k][2].y, r[k][2].z};
            own.ikn = r[k][1].w;
            own.ikt = r[k][2].w;
        }
    }
}
__device__ __forceinline__ float4 lam4(const Contact<float> &c) { return make_float4(c.lam.x, c.lam.y, c.lam.z, 0.0f); }
__device__ __forceinline__ float4 lam4a(const Contact<F2> &c) { return make_float4(c.lam.x.x, c.lam.y.x, c.lam.z.x, 0.0f); }
__device__ __forceinline__ float4 lam4b(const Contact<F2> &c) { return make_float4(c.lam.x.y, c.lam.y.y, c.lam.z.y, 0.0f); }

// One substep of one environment (the arithmetic of step_kernel.cuh, contacts in the
// same order: link, then sphere), its contact records written at sp.rec.
// With TAPE the impulses after every iteration and the iteration sums are
// recorded in the slot's current tape block; with PADS the pad forces of the
// substep are added to S.padacc; with replay_nc >= 0 the substep's records
// at sp.rec are those of an earlier run from the same state (replay_nc
// contacts, setup included), which replaces the enumeration and the setup.
// Returns the contact count (0 on overflow). Not inlined, with the flags as
// arguments: one copy serves every pass. (The iterations' arithmetic has a fixed
// contraction, contact.cuh, so a recorded tape is bit for bit the forward's.)
template <int GW>
__device__ __noinline__ int fwd_substep(const AdjArgs &a, const Env &E_, Body &b, const float4 *L0,
                                        const float4 *L1, const SlotPtr &sp_, GroupSm<GW> &S, const PadTable &PT,
                                        const AGroup<GW> &G_, int &parity_, int &st_, int tape_flag,
                                        int pads_flag, int replay_nc) {
    const bool TAPE = tape_flag != 0, PADS = pads_flag != 0;
    // by-value copies of what the loops read: through the references every
    // store to the tape or to shared memory could alias them and force reloads
    const Env E = E_;
    const SlotPtr sp = sp_;
    const AGroup<GW> G = G_;
    int parity = parity_, st = st_;
    constexpr int T = AGroup<GW>::T;
    const DevScene sc = a.sc;   // by value, as E below
    const DevConfig cfg = a.cfg;
    const int Lk = sc.n_links, P = sc.n_pads, cap = cfg.c_max;
    const float h = cfg.h, inv_h = 1.0f / h, inv_L = 1.0f / sc.link_len;
    const V3 grav = mk(cfg.gx * h, cfg.gy * h, cfg.gz * h);
    const V3 v_pred = b.v + grav;
    const V3 w_pred = b.w;
    const M3 R = qmat(b.q);
    const S6 Wi = world_inv_inertia_f(R, E.Jb, E.inv_m);
    const int lane = G.lane, gt = G.gt;

    int nc = 0;
    const bool replay = replay_nc >= 0;
    if (replay) {
        // the records this substep's first run left, setup included: no
        // enumeration (the run is deterministic, so they are its own)
        nc = replay_nc;
    } else {
        // contact enumeration, in the step's order (link, then sphere): sphere and
        // cluster centres to world, the (link, cluster) cull by the clusters' enclosing
        // spheres, then a thread tests the eight spheres of a surviving pair
        const int ncl = (E.NS + kCluster - 1) / kCluster;
        const float inv_ncl = 1.0f / (float)ncl;
        G.sync();   // (a reverse sweep may just have read the ring in the centres' place)
#pragma unroll 1
        for (int j = gt; j < ncl * kCluster; j += T) {
            float4 o = make_float4(kFar, kFar, kFar, 0.0f);   // (padding of the last cluster: far away)
            if (j < E.NS) {
                const float4 s4 = __ldg(sc.spheres + E.sfirst + j);
                const V3 cr = mmul(R, xyz(s4));
                o = make_float4(cr.x, cr.y, cr.z, s4.w);
            }
            S.en.sph[(j >> 3) * kSphStride + (j & 7)] = o;
        }
#pragma unroll 1
        for (int k = gt; k < ncl; k += T) {
            const float4 cl = __ldg(sc.clusters + E.cfirst + k);
            const V3 cr = mmul(R, xyz(cl));
            S.en.clc[k] = make_float4(cr.x, cr.y, cr.z, cl.w);
        }
#pragma unroll 1
        for (int l = gt; l < Lk; l += T) {
            const V3 xa = b.x - xyz(__ldg(L0 + l * kLinkStride));
            S.xa[l] = make_float4(xa.x, xa.y, xa.z, 0.0f);
            S.ax[l] = __ldg(L0 + l * kLinkStride + 1);
            S.lbeg[l] = 0;
            S.lend[l] = 0;
        }
        G.sync();
        const int ncp = Lk * ncl;
        int nclp = 0;
#pragma unroll 1
        for (int p0 = 0; p0 < ncp; p0 += T) {
            const int p = p0 + gt;
            bool keep = false;
            int e = 0;
            if (p < ncp) {
                const int l = min((int)(((float)p + 0.5f) * inv_ncl), Lk - 1), k = p - l * ncl;
                const float4 cc = S.en.clc[k];
                keep = cluster_reaches(sc, cfg, l, xyz(S.xa[l]) + xyz(cc), cc.w, xyz(S.ax[l]));
                e = (l << 8) | k;
            }
            const int off = gcompact<GW, 1>(keep, nclp, G, S, parity);
            if (keep) S.en.clp[off] = (unsigned short)e;
        }
        G.sync();
#pragma unroll 1
        for (int e0 = 0; e0 < nclp; e0 += T) {
            unsigned hits = 0;
            int e = 0;
            if (e0 + gt < nclp) {
                e = S.en.clp[e0 + gt];
                const int l = e >> 8, k = e & 0xff;
                hits = cluster_hits(sc, cfg, l, k, xyz(S.xa[l]), xyz(S.ax[l]), S.en.sph + k * kSphStride, E.NS, inv_L);
            }
            const int idx = gcompact<GW, 4>(__popc(hits), nc, G, S, parity);
            const int cj = (e & 0xff00) | ((e & 0xff) * kCluster);
#pragma unroll
            for (int i = 0; i < kCluster; ++i) {
                const int at = idx + __popc(hits & ((1u << i) - 1u));
                if (((hits >> i) & 1u) && at < cap) S.clist[at] = (unsigned short)(cj + i);
            }
        }
        G.sync();
        if (nc > cap) {   // more contacts than the per-env capacity: as the step, no contacts
            st |= IH_ENV_OVERFLOW;
            nc = 0;
        }
    }

    // contact setup by the contact's thread (or its results from the records); a
    // block of four warps keeps its one contact a thread in registers
    const float trW = Wi.xx + Wi.yy + Wi.zz;
    Contact<float> own;
    own.clear();
    if (replay) {
        load_constants<GW, false>(sp, S, G, nc, own);
        if (GW == 1)
#pragma unroll 1
            for (int ci = kRC + gt; ci < nc; ci += T) sp.lamf[ci] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    } else {
        if (GW == 1)   // empty slots up to the next whole pair of slots
#pragma unroll 1
            for (int k = nc >> 5; k < 4 && k <= ((nc - 1) >> 5 | 1); ++k)
                if (lane + 32 * k >= nc) cp_store(S, k, lane, mk(0, 0, 0), mk(0, 0, 1), mk(0, 0, 0), 0.0f, 0.0f);
#pragma unroll 1
        for (int ci = gt; ci < nc; ci += T) {
            float4 *rc = sp.rec + 4 * ci;
            const int e = S.clist[ci], l = e >> 8, j = e & 0xff;
            const int e0 = ci > 0 ? S.clist[ci - 1] >> 8 : -1, e1 = ci < nc - 1 ? S.clist[ci + 1] >> 8 : -1;
            if (e0 != l) S.lbeg[l] = (unsigned short)ci;
            if (e1 != l) S.lend[l] = (unsigned short)(ci + 1);
            const float4 s4 = S.en.sph[(j >> 3) * kSphStride + (j & 7)];
            const V3 cr = xyz(s4);
            const Hit hh = hit_link(sc, l, xyz(S.xa[l]) + cr, s4.w, xyz(S.ax[l]), L0, inv_L);
            const V3 r = cr - hh.n * s4.w;
            const unsigned char pad = PT.find(l, hh.t);
            S.cpad[ci] = pad;
            const CSetup cs = setup_contact(r, hh.n, hh.gap, l, Wi, trW, E.inv_m, cfg, L0, L1, b.x, inv_h);
            rc[0] = make_float4(r.x, r.y, r.z, hh.gap);
            rc[1] = make_float4(hh.n.x, hh.n.y, hh.n.z, cs.ikn);
            rc[2] = make_float4(cs.cc.x, cs.cc.y, cs.cc.z, cs.ikt);
            rc[3] = make_float4(hh.t, __int_as_float(l | (pad << 8)), __int_as_float(j), 0.0f);
            if (ci >= kRC) {
                if (GW == 1) sp.lamf[ci] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);   // a further contact: its impulse in memory
            } else if constexpr (GW == 1) {
                cp_store(S, ci >> 5, lane, r, hh.n, cs.cc, cs.ikn, cs.ikt);
            } else {
                own.r = {r.x, r.y, r.z};
                own.n = {hh.n.x, hh.n.y, hh.n.z};
                own.c = {cs.cc.x, cs.cc.y, cs.cc.z};
                own.ikn = cs.ikn;
                own.ikt = cs.ikt;
            }
        }
    }
    G.sync();

    // Jacobi projected-impulse iterations, on the warps that hold contacts
    V3 vv = v_pred, ww = w_pred;
    if (nc > 0) {
        const int aw = GW == 1 ? 1 : min(kWarps<GW>, (nc + 31) >> 5);
        const float inv_nc = 1.0f / (float)nc, mu_s = 4096.0f * E.mu;
        auto add1 = [&](float (&acc)[6], const Contact<float> &c) {
            float s[6];
            c.wrench(s);
#pragma unroll
            for (int q = 0; q < 6; ++q) acc[q] += s[q];
        };
        auto add2 = [&](float (&acc)[6], const Contact<F2> &c) {
            F2 s[6];
            c.wrench(s);
#pragma unroll
            for (int q = 0; q < 6; ++q) acc[q] = (acc[q] + s[q].x) + s[q].y;
        };
        // the impulse of register slot k after iteration it, to the tape
        auto tape = [&](int it, int k, float4 lam) {
            const int ci = gt + T * k;
            store_if(TAPE && ci < nc, sp.lamh + (size_t)it * cap + ci, lam);
        };
        auto further = [&](int it, float (&acc)[6]) {   // contacts kRC, ... in the same per-thread order
#pragma unroll 1
            for (int ci = kRC + gt; ci < nc; ci += T) {
                const float4 *rc = sp.rec + 4 * ci;
                const float4 r0 = rc[0], r1 = rc[1], r2 = rc[2], l4 = sp.lamf[ci];
                Contact<float> c;
                c.r = {r0.x, r0.y, r0.z};
                c.n = {r1.x, r1.y, r1.z};
                c.c = {r2.x, r2.y, r2.z};
                c.lam = {l4.x, l4.y, l4.z};
                c.ikn = r1.w;
                c.ikt = r2.w;
                c.update(vv, ww, mu_s, inv_nc);
                sp.lamf[ci] = lam4(c);
                add1(acc, c);
                if (TAPE) sp.lamh[(size_t)it * cap + ci] = lam4(c);
            }
        };
        auto body = [&](int it, float (&acc)[6], auto one) {
            if constexpr (GW == 1 || decltype(one)::value) width_sum6<32>(acc, kFull, lane);
            else gsum6<GW>(acc, G, S, parity, aw);
            float4 *q = reinterpret_cast<float4 *>(sp.sh + 8 * it);
            store_if(TAPE && gt == 0, q, make_float4(acc[0], acc[1], acc[2], acc[3]));
            store_if(TAPE && gt == 0, q + 1, make_float4(acc[4], acc[5], 0.0f, 0.0f));
            vv = v_pred + mk(acc[0], acc[1], acc[2]) * E.inv_m;
            ww = w_pred + smul(Wi, mk(acc[3], acc[4], acc[5]));
        };
        // one loop per number of occupied slots, each a straight stretch of code
        auto last = [&](int k, float4 lam) {
            const int ci = gt + T * k;
            if (ci < nc) S.clam[ci] = lam;
        };
        if constexpr (GW == 1) {
            const Vec<F2> z2 = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
            const Vec<float> z1 = {0.0f, 0.0f, 0.0f};
            if (nc <= 32) {
                Contact<float> c0;
                cp_load(S, 0, lane, c0);
                c0.lam = z1;
#pragma unroll 1
                for (int it = 0; it < E.iters; ++it) {
                    float acc[6] = {0, 0, 0, 0, 0, 0};
                    c0.update(vv, ww, mu_s, inv_nc);
                    add1(acc, c0);
                    tape(it, 0, lam4(c0));
                    body(it, acc, Flag<true>{});
                }
                last(0, lam4(c0));
            } else if (nc <= 64) {
                Contact<F2> c0;
                cp_load(S, 0, lane, c0);
                c0.lam = z2;
#pragma unroll 1
                for (int it = 0; it < E.iters; ++it) {
                    float acc[6] = {0, 0, 0, 0, 0, 0};
                    c0.update(vv, ww, mu_s, inv_nc);
                    add2(acc, c0);
                    tape(it, 0, lam4a(c0));
                    tape(it, 1, lam4b(c0));
                    body(it, acc, Flag<true>{});
                }
                last(0, lam4a(c0));
                last(1, lam4b(c0));
            } else if (nc <= 96) {
                Contact<F2> c0;
                Contact<float> c2;
                cp_load(S, 0, lane, c0);
                cp_load(S, 2, lane, c2);
                c0.lam = z2;
                c2.lam = z1;
#pragma unroll 1
                for (int it = 0; it < E.iters; ++it) {
                    float acc[6] = {0, 0, 0, 0, 0, 0};
                    c0.update(vv, ww, mu_s, inv_nc);
                    c2.update(vv, ww, mu_s, inv_nc);
                    add2(acc, c0);
                    add1(acc, c2);
                    tape(it, 0, lam4a(c0));
                    tape(it, 1, lam4b(c0));
                    tape(it, 2, lam4(c2));
                    body(it, acc, Flag<true>{});
                }
                last(0, lam4a(c0));
                last(1, lam4b(c0));
                last(2, lam4(c2));
            } else {
                Contact<F2> c0, c2;
                cp_load(S, 0, lane, c0);
                cp_load(S, 2, lane, c2);
                c0.lam = z2;
                c2.lam = z2;
#pragma unroll 1
                for (int it = 0; it < E.iters; ++it) {
                    float acc[6] = {0, 0, 0, 0, 0, 0};
                    c0.update(vv, ww, mu_s, inv_nc);
                    c2.update(vv, ww, mu_s, inv_nc);
                    add2(acc, c0);
                    add2(acc, c2);
                    tape(it, 0, lam4a(c0));
                    tape(it, 1, lam4b(c0));
                    tape(it, 2, lam4a(c2));
                    tape(it, 3, lam4b(c2));
                    further(it, acc);
                    body(it, acc, Flag<true>{});
                }
                last(0, lam4a(c0));
                last(1, lam4b(c0));
                last(2, lam4a(c2));
                last(3, lam4b(c2));
            }
        } else {
            // (more: two contacts a thread, side by side)
            auto iterate = [&](auto one, auto more, Contact<float> &own2) {
#pragma unroll 1
                for (int it = 0; it < E.iters; ++it) {
                    float acc[6] = {0, 0, 0, 0, 0, 0};
                    own.update(vv, ww, mu_s, inv_nc);
                    if constexpr (decltype(more)::value) own2.update(vv, ww, mu_s, inv_nc);
                    add1(acc, own);
                    if constexpr (decltype(more)::value) add1(acc, own2);
                    tape(it, 0, lam4(own));
                    if constexpr (decltype(more)::value) tape(it, 1, lam4(own2));
                    body(it, acc, one);
                }
                last(0, lam4(own));
                if constexpr (decltype(more)::value)
                    if (gt + T < nc) sp.lamf[gt + T] = lam4(own2);
            };
            if (aw == 1) {
                if (G.wg == 0) iterate(Flag<true>{}, Flag<false>{}, own);
            } else if (GW != kTwo || nc <= kRC) {
                if (G.wg < aw) iterate(Flag<false>{}, Flag<false>{}, own);
            } else if constexpr (GW == kTwo) {
                Contact<float> own2;
                load_second<GW>(sp, G, nc, own2);   // (its record is this thread's own)
                iterate(Flag<false>{}, Flag<true>{}, own2);
            }
            if (aw < kWarps<GW>) {   // the body's velocity to the other warps
                if (gt == 0) {
                    S.fin[0] = vv.x; S.fin[1] = vv.y; S.fin[2] = vv.z;
                    S.fin[3] = ww.x; S.fin[4] = ww.y; S.fin[5] = ww.z;
                }
                G.sync();
                vv = mk(S.fin[0], S.fin[1], S.fin[2]);
                ww = mk(S.fin[3], S.fin[4], S.fin[5]);
                parity = 0;   // (the warps have used the reduction's buffers differently often)
            }
        }
    }
    b.v = vv;
    b.w = ww;
    b.x = b.x + b.v * h;
    {
        const float wn = sqrtf(dot(b.w, b.w));
        float sn, cs;
        sincosf(0.5f * wn * h, &sn, &cs);
        const float kq = (wn > 0.0f) ? sn / wn : 0.5f * h;
        b.q = qnorm(qmul_f({cs, b.w.x * kq, b.w.y * kq, b.w.z * kq}, b.q));
    }
    G.sync();
    if (PADS) {
        // pad forces -lambda / h, each pad summing the contacts of its link in
        // order, one thread per pad and component (never on a replayed substep)
#pragma unroll 1
        for (int k = gt; k < 3 * P; k += T) {
            const int p = k / 3, comp = k - 3 * p;
            const int l = __ldg(sc.pad_link + p);
            float f = 0.0f;
            const int e = nc > 0 ? S.lend[l] : 0, es = min(e, kRC);
            int ci = S.lbeg[l];
            const float *lc = reinterpret_cast<const float *>(S.clam) + comp;
#pragma unroll 4
            for (; ci < es; ++ci) f -= (S.cpad[ci] == p ? lc[4 * ci] : 0.0f) * inv_h;
#pragma unroll 1
            for (; ci < e; ++ci) f -= (S.cpad[ci] == p ? reinterpret_cast<const float *>(sp.lamf + ci)[comp] : 0.0f) * inv_h;
            S.padacc[k] += f;
        }
    }
    G.sync();
    parity_ = parity;
    st_ = st;
    return nc;
}

// d bias / d gap (contact_bias: gap / h when separated, else the clamped
// Baumgarte term)
__device__ __forceinline__ float bias_slope(const DevConfig &cfg, float gap) {
    if (gap > 0.0f) return 1.0f / cfg.h;
    const float z = gap + cfg.slop;
    if (!(z < 0.0f)) return 0.0f;
    return (cfg.beta * z / cfg.h > -cfg.vmax) ? cfg.beta / cfg.h : 0.0f;
}

// The reverse sweep's smoothing functions use the hardware's approximate
// exponential, reciprocal and reciprocal square root (a few ulp each): they
// sit at the head of every reverse iteration's dependent chain, and their
// error is far inside the gradient's tolerance against the FP64 adjoint.
__device__ __forceinline__ float sigmoid(float x) { return __fdividef(1.0f, 1.0f + __expf(-x)); }

// Reverse of the smoothed radial clamp out = z smin(|z|, L) / |z| for the
// incoming derivative g: dL/dz = g ra + zh (zh . g) pr and dL/dL = (zh . g) pb,
// the four factors formed here from z and L alone. At z = 0 exactly (and below
// 1e-15, where the expressions leave FP32's range) the derivative of the exact
// clamp inside the disk (identity) is used. With
// Q = sqrt((a - L)^2 + (w L)^2), smin(a, L) = (a + L - Q) / 2 is evaluated as
// L (4a - w^2 L) / (2 (a + L + Q)), the same value without the cancellation
// of a + L - Q when the clamp does not bind (a << L).
__device__ __forceinline__ void disk_factors(float a2, float L, float w, float &ia, float &ra, float &pr, float &pb) {
    const bool at0 = !(a2 > 1e-30f);
    const float r = rsqrt_ftz(at0 ? 1.0f : a2);
    const float a = (at0 ? 1.0f : a2) * r;
    const float dl = a - L, wL = w * L;
    const float Q2 = fmaxf(fmaf(dl, dl, wL * wL), 1e-37f);
    const float iQ = rsqrt_ftz(Q2);
    const float phi = __fdividef(L * fmaf(-w, wL, 4.0f * a), 2.0f * fmaf(Q2, iQ, a + L));
    const float k = dl * iQ;
    ia = at0 ? 0.0f : r;
    ra = at0 ? (L > 0.0f ? 1.0f : 0.0f) : phi * r;
    pr = at0 ? 0.0f : fmaf(-0.5f, k, 0.5f) - phi * r;
    pb = at0 ? 0.0f : fmaf(0.5f, k - w * wL * iQ, 0.5f);
}
__device__ __forceinline__ void disk_factors(F2 a2, F2 L, float w, F2 &ia, F2 &ra, F2 &pr, F2 &pb) {
    disk_factors(a2.x, L.x, w, ia.x, ra.x, pr.x, pb.x);
    disk_factors(a2.y, L.y, w, ia.y, ra.y, pr.y, pb.y);
}
__device__ __forceinline__ F2 sigmoid(F2 x) { return make_float2(sigmoid(x.x), sigmoid(x.y)); }
__device__ __forceinline__ float t_sum(float a) { return a; }
__device__ __forceinline__ float t_sum(F2 a) { return a.x + a.y; }

// Reverse of the narrowphase (hit_box_local / hit_capsule) for the sphere centred
// at x + cr: the derivative w.r.t. the centre given those w.r.t. gap and n.
__device__ __forceinline__ V3 hit_bwd(const DevScene &sc, int l, V3 x, V3 cr, const float4 *L0, float gb, V3 nb) {
    const float4 A0 = __ldg(L0 + l * kLinkStride);
    const float4 Aq = __ldg(L0 + l * kLinkStride + 2);
    const Q4 q = {Aq.x, Aq.y, Aq.z, Aq.w};
    if (l == 0) {
        const float hx = sc.palm_hx, hy = sc.palm_hy, hz = sc.palm_hz;
        const V3 cl = qrot_inv(q, (x + cr) - xyz(A0));
        const V3 k = mk(fminf(fmaxf(cl.x, -hx), hx), fminf(fmaxf(cl.y, -hy), hy), fminf(fmaxf(cl.z, -hz), hz));
        V3 clb = mk(0, 0, 0);
        if (!((k.x == cl.x) && (k.y == cl.y) && (k.z == cl.z))) {
            const V3 d = cl - k;
            const float inv = rsqrtf(dot(d, d));
            const V3 nl = d * inv;
            const V3 nlb = qrot_inv(q, nb);
            const V3 db = (nlb - nl * dot(nl, nlb)) * inv + nl * gb;
            clb = mk(k.x != cl.x ? db.x : 0.0f, k.y != cl.y ? db.y : 0.0f, k.z != cl.z ? db.z : 0.0f);
        } else {   // the face hit_box_local chose; the normal is constant, gap = +-cl_axis - half - r
            float best = hx - cl.x;
            int face = 0;
            if (hx + cl.x < best) { best = hx + cl.x; face = 1; }
            if (hy - cl.y < best) { best = hy - cl.y; face = 2; }
            if (hy + cl.y < best) { best = hy + cl.y; face = 3; }
            if (hz - cl.z < best) { best = hz - cl.z; face = 4; }
            if (hz + cl.z < best) { best = hz + cl.z; face = 5; }
            const float g = (face & 1) ? -gb : gb;
            clb = mk(face >> 1 == 0 ? g : 0.0f, face >> 1 == 1 ? g : 0.0f, face >> 1 == 2 ? g : 0.0f);
        }
        return qrot(q, clb);
    }
    const V3 ca = (x - xyz(A0)) + cr;
    const V3 d = xyz(__ldg(L0 + l * kLinkStride + 1));
    const float tr = dot(ca, d) * (1.0f / sc.link_len);
    const float t = fminf(fmaxf(tr, 0.0f), 1.0f);
    const V3 diff = ca - d * (t * sc.link_len);
    const float d2 = dot(diff, diff);
    if (d2 < 1e-18f) return mk(0, 0, 0);   // centre on the axis: constant normal and gap
    const float inv = rsqrtf(d2);
    const V3 n = diff * inv;
    V3 db = (nb - n * dot(n, nb)) * inv + n * gb;
    if (tr > 0.0f && tr < 1.0f) db = db - d * dot(d, db);   // t follows the centre inside the segment
    return db;
}

__device__ __forceinline__ void outer_add(float (&M)[9], V3 a, V3 b, float s) {
    const float av[3] = {a.x * s, a.y * s, a.z * s}, bv[3] = {b.x, b.y, b.z};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) M[3 * i + j] += av[i] * bv[j];
}

// Reverse of one contact's setup and narrowphase (lever arm r, normal n, gap, 1/k_n,
// 1/k_t, link l, sphere j) given the derivatives w.r.t. its constants
// nb, rb, cb, iknb, iktb: the thread's parts of d/dx, d/d(1/m), d/dW and d/dR
// accumulate.
__device__ __forceinline__ void contact_setup_bwd(V3 r, V3 n, float gap, float ikn, float ikt, int l, int j, V3 nb, V3 rb, V3 cb,
                                                  float iknb, float iktb,
                                                  const S6 &Wi, float trW, const M3 &R, V3 x, int sfirst,
                                                  const DevScene &sc, const DevConfig &cfg, const float4 *L0,
                                                  const float4 *L1, float inv_h, float (&Wbar)[9], float (&Rbar)[9],
                                                  V3 &xb_l, float &invm_l) {
    // 1/k_n and 1/k_t = 2 / (tr K - k_n)
    float knb = -iknb * ikn * ikn;
    const float Db = -iktb * ikt * ikt * 0.5f;
    const float trKb = Db;
    knb -= Db;
    // k_n = 1/m + (r x n) . W (r x n)
    const V3 rn = cross(r, n);
    const V3 rnb = smul(Wi, rn) * (2.0f * knb);
    invm_l += knb + 3.0f * trKb;
    outer_add(Wbar, rn, rn, knb);
    rb = rb + cross(n, rnb);
    nb = nb + cross(rnb, r);
    // tr K = 3/m + |r|^2 tr W - r . W r
    rb = rb + (r * (2.0f * trW) - smul(Wi, r) * 2.0f) * trKb;
    const float rr = dot(r, r) * trKb;
    Wbar[0] += rr; Wbar[4] += rr; Wbar[8] += rr;
    outer_add(Wbar, r, r, -trKb);
    // c = v_link - n b(gap)
    const float bias = contact_bias(cfg, gap);
    const float gb = -dot(n, cb) * bias_slope(cfg, gap);
    nb = nb - cb * bias;
    if (l != 0) {   // v_link = (T_end T_start^-1 p - p) / h, p = x + r
        const float4 Aq = __ldg(L0 + l * kLinkStride + 2), Bq = __ldg(L1 + l * kLinkStride + 2);
        const Q4 qa = {Aq.x, Aq.y, Aq.z, Aq.w}, qe = {Bq.x, Bq.y, Bq.z, Bq.w};
        const V3 yb = (qrot(qa, qrot_inv(qe, cb)) - cb) * inv_h;
        xb_l = xb_l + yb;
        rb = rb + yb;
    }
    // r = R s_j - n r_j, gap and n from the sphere centre x + R s_j
    const float4 s4 = __ldg(sc.spheres + sfirst + j);
    nb = nb - rb * s4.w;
    const V3 cr = mmul(R, xyz(s4));
    const V3 hb = hit_bwd(sc, l, x, cr, L0, gb, nb);
    xb_l = xb_l + hb;
    outer_add(Rbar, rb + hb, xyz(s4), 1.0f);
}

// The reverse of one contact's (T = float) or two contacts' (float2, packed) updates
// in the Jacobi iterations: the derivative lb w.r.t. the impulse after the current
// iteration and those w.r.t. the constants r, n, c, 1/k_n, 1/k_t, accumulated.
// a x b added to s
template <typename T>
__device__ __forceinline__ Vec<T> t_cross_add(const Vec<T> &a, const Vec<T> &b, const Vec<T> &s) {
    return {t_fma(a.y, b.z, t_fma(t_neg(a.z), b.y, s.x)), t_fma(a.z, b.x, t_fma(t_neg(a.x), b.z, s.y)),
            t_fma(a.x, b.y, t_fma(t_neg(a.y), b.x, s.z))};
}
template <typename T>
__device__ __forceinline__ Vec<T> t_vec(V3 v) { return {t_all<T>(v.x), t_all<T>(v.y), t_all<T>(v.z)}; }
template <typename T>
__device__ __forceinline__ Vec<T> t_axpy(T k, const Vec<T> &a, const Vec<T> &s) {
    return {t_fma(k, a.x, s.x), t_fma(k, a.y, s.y), t_fma(k, a.z, s.z)};
}
template <typename T>
__device__ __forceinline__ Vec<T> t_scale(T k, const Vec<T> &a) { return {t_mul(k, a.x), t_mul(k, a.y), t_mul(k, a.z)}; }

// What the reverse of an update takes from the forward alone: u, un = u . n, lo =
// lambda . n, the normal impulse ln and the clamps' derivatives (disk_factors, and
// sig, the normal clamp's). No derivative enters, so they are formed an iteration
// ahead, in the shadow of the reduction.
template <typename T>
struct Factors {
    Vec<T> u, zh;
    T un, lo, ln, ra, pr, pb, sig;
    // c holds the constants and the impulse before the iteration
    __device__ __forceinline__ void form(const Contact<T> &c, V3 Vi, V3 Wv, float mu, float width, float beta_s) {
        const Vec<T> tW = t_vec<T>(Wv), tV = t_vec<T>(Vi);
        u = t_cross_add(tW, c.r, Vec<T>{t_fma(c.c.x, t_all<T>(-1.0f), tV.x), t_fma(c.c.y, t_all<T>(-1.0f), tV.y),
                                        t_fma(c.c.z, t_all<T>(-1.0f), tV.z)});
        un = t_dot(u, c.n);
        lo = t_dot(c.lam, c.n);
        const T nun = t_neg(un), zn = t_fma(nun, c.ikn, lo);
        ln = t_relu(zn);
        const Vec<T> zt = t_axpy(t_neg(c.ikt), t_axpy(nun, c.n, u), t_axpy(t_neg(lo), c.n, c.lam));
        T ia;
        disk_factors(t_dot(zt, zt), t_mul(t_all<T>(mu), ln), width, ia, ra, pr, pb);
        zh = t_scale(ia, zt);
        sig = sigmoid(t_mul(t_all<T>(beta_s), zn));
    }
};

template <typename T>
struct ContactBwd {
    Vec<T> lb, nb, rb, cb;
    T iknb, iktb, mub;
    __device__ __forceinline__ void clear() {
        const T o = t_all<T>(0.0f);
        lb = nb = rb = cb = {o, o, o};
        iknb = iktb = mub = o;
    }
    // One iteration: c holds the constants and the impulse before it, f its factors,
    // l1 the impulse after it; vm = Vb / m and g = W Wb of the derivatives Vb, Wb
    // w.r.t. the body's velocity after it, Wv the angular velocity before it. Adds the
    // derivatives w.r.t. that velocity to acc. (An empty slot adds zeros: its 1/k and
    // r are zero.)
    __device__ __forceinline__ void step(const Contact<T> &c, const Factors<T> &f, const Vec<T> &l1, V3 vm, V3 g, V3 Wv, float mu,
                                         float inv_nc, T (&acc)[6]) {
        const Vec<T> tg = t_vec<T>(g), tW = t_vec<T>(Wv);
        // V and W after the iteration: the impulse's share
        lb = t_cross_add(tg, c.r, Vec<T>{t_add(lb.x, t_all<T>(vm.x)), t_add(lb.y, t_all<T>(vm.y)), t_add(lb.z, t_all<T>(vm.z))});
        rb = t_cross_add(l1, tg, rb);
        // lambda' = lambda + (n ln + lt - lambda) / n_c
        const Vec<T> lpb = t_scale(t_all<T>(inv_nc), lb);
        lb = t_scale(t_all<T>(1.0f - inv_nc), lb);
        const T s = t_dot(f.zh, lpb), Lb = t_mul(s, f.pb), nun = t_neg(f.un), nlo = t_neg(f.lo);
        const Vec<T> ztb = t_axpy(t_mul(s, f.pr), f.zh, t_scale(f.ra, lpb));
        mub = t_fma(f.ln, Lb, mub);
        const T znb = t_mul(t_fma(t_all<T>(mu), Lb, t_dot(c.n, lpb)), f.sig);
        const T nzt = t_dot(c.n, ztb);
        iknb = t_fma(znb, nun, iknb);
        // (u - n un) . ztb
        iktb = t_fma(t_all<T>(-1.0f), t_fma(nun, nzt, t_dot(f.u, ztb)), iktb);
        const T unb = t_fma(c.ikt, nzt, t_neg(t_mul(znb, c.ikn))), lob = t_fma(t_all<T>(-1.0f), nzt, znb);
        const Vec<T> ub = t_axpy(unb, c.n, t_scale(t_neg(c.ikt), ztb));
        // u = V + W x r - c
        acc[0] = t_add(acc[0], ub.x); acc[1] = t_add(acc[1], ub.y); acc[2] = t_add(acc[2], ub.z);
        const Vec<T> m = t_cross_add(c.r, ub, Vec<T>{acc[3], acc[4], acc[5]});
        acc[3] = m.x; acc[4] = m.y; acc[5] = m.z;
        nb = t_axpy(f.ln, lpb, nb);
        nb = t_axpy(t_fma(c.ikt, f.un, nlo), ztb, nb);
        nb = t_axpy(lob, c.lam, nb);
        nb = t_axpy(unb, f.u, nb);
        lb = t_axpy(lob, c.n, Vec<T>{t_add(lb.x, ztb.x), t_add(lb.y, ztb.y), t_add(lb.z, ztb.z)});
        rb = t_cross_add(ub, tW, rb);
        cb = {t_fma(ub.x, t_all<T>(-1.0f), cb.x), t_fma(ub.y, t_all<T>(-1.0f), cb.y), t_fma(ub.z, t_all<T>(-1.0f), cb.z)};
    }
};

// The reverse iterations of the register-resident contacts of a thread: units U0
// (slots 0, or 0 and 1) and U1 (slots 2, or 2 and 3; NoUnit when absent), and the
// contacts past kRC from memory.
// Vb, Wb enter as the derivatives w.r.t. the velocity after the last iteration and
// leave as those before the first; vpb, wpb, Wbar, invm_l accumulate.
struct NoUnit {};
template <int GW>
struct RevCtx {
    const SlotPtr &sp;
    GroupSm<GW> &S;
    const AGroup<GW> &G;
    const S6 &Wi;
    V3 v_pred, w_pred;
    float inv_m, mu, inv_nc, width, beta_s;
    int cap, nc, I, aw, n_pads;
};
__device__ __forceinline__ void set_half(Vec<float> &v, int, float4 l) { v = {l.x, l.y, l.z}; }
__device__ __forceinline__ void set_half(Vec<F2> &v, int h, float4 l) {
    if (h == 0) { v.x.x = l.x; v.y.x = l.y; v.z.x = l.z; }
    else { v.x.y = l.x; v.y.y = l.y; v.z.y = l.z; }
}
__device__ __forceinline__ V3 get_half(const Vec<float> &v, int) { return mk(v.x, v.y, v.z); }
__device__ __forceinline__ V3 get_half(const Vec<F2> &v, int h) { return h == 0 ? mk(v.x.x, v.y.x, v.z.x) : mk(v.x.y, v.y.y, v.z.y); }
__device__ __forceinline__ float get_half(float v, int) { return v; }
__device__ __forceinline__ float get_half(F2 v, int h) { return h == 0 ? v.x : v.y; }

// one unit: its reverse state, its impulses after iterations it and it - 1, and,
// when AHEAD, the factors of iteration it, formed an iteration early
template <int GW, typename T>
struct RevUnit {
    static constexpr int N = sizeof(T) / sizeof(float);
    ContactBwd<T> b;
    Factors<T> f;
    Vec<T> l1, l0;
    int slot;
    __device__ __forceinline__ void init(const RevCtx<GW> &x, int slot_) {
        slot = slot_;
        b.clear();
#pragma unroll
        for (int h = 0; h < N; ++h) {
            const int ci = x.G.gt + AGroup<GW>::T * (slot + h);
            float4 f4 = make_float4(0, 0, 0, 0), l4 = f4;
            if (ci < x.nc) {   // the pad's derivative on the contact's final impulse
                const int pad = rec_pad(kHeld<GW> == kRC || ci < kRC ? x.S.meta[ci] : x.sp.rec[4 * ci + 3]);
                if (pad < x.n_pads) f4 = make_float4(-x.S.fbar[3 * pad], -x.S.fbar[3 * pad + 1], -x.S.fbar[3 * pad + 2], 0.0f);
                l4 = x.sp.lamh[(size_t)(x.I - 1) * x.cap + ci];
            }
            set_half(b.lb, h, f4);
            set_half(l1, h, l4);
        }
    }
    // the impulses after iteration it: their copy (zeros before the first and in empty
    // slots), and their values once it has arrived
    __device__ __forceinline__ void request(const RevCtx<GW> &x, int it) const {
#pragma unroll
        for (int h = 0; h < N; ++h) {
            const int ci = x.G.gt + AGroup<GW>::T * (slot + h);
            copy_async(&x.S.ring[it & (kRing - 1)][ci], x.sp.lamh + (size_t)max(it, 0) * x.cap + min(ci, x.nc - 1),
                       it >= 0 && ci < x.nc ? 16 : 0);
        }
    }
    __device__ __forceinline__ void arrived(const RevCtx<GW> &x, int it, Vec<T> &v) const {
#pragma unroll
        for (int h = 0; h < N; ++h) set_half(v, h, x.S.ring[it & (kRing - 1)][x.G.gt + AGroup<GW>::T * (slot + h)]);
    }
    __device__ __forceinline__ void constants(const RevCtx<GW> &x, const Contact<float> &own, Contact<T> &c) const {
        if constexpr (GW == 1) cp_load(x.S, slot, x.G.lane, c);
        else c = own;
        c.lam = l0;
    }
    __device__ __forceinline__ void form(const RevCtx<GW> &x, const Contact<float> &own, int it, V3 Vi, V3 Wv) {   // of iteration it
        arrived(x, it - 1, l0);
        Contact<T> c;
        constants(x, own, c);
        f.form(c, Vi, Wv, x.mu, x.width, x.beta_s);
    }
    __device__ __forceinline__ void step(const RevCtx<GW> &x, const Contact<float> &own, V3 vm, V3 g, V3 Wv, float (&acc)[6]) {
        Contact<T> c;
        constants(x, own, c);
        const T o = t_all<T>(0.0f);
        T s[6] = {o, o, o, o, o, o};
        b.step(c, f, l1, vm, g, Wv, x.mu, x.inv_nc, s);
#pragma unroll
        for (int q = 0; q < 6; ++q) acc[q] += t_sum(s[q]);
        l1 = l0;
    }
    // ... of a thread's second contact (four warps), straight onto the thread's sums
    __device__ __forceinline__ void step_on(const RevCtx<GW> &x, const Contact<float> &own, V3 vm, V3 g, V3 Wv, float (&acc)[6]) {
        Contact<T> c;
        constants(x, own, c);
        b.step(c, f, l1, vm, g, Wv, x.mu, x.inv_nc, acc);
        l1 = l0;
    }
    // the derivatives w.r.t. the constants, in the ring's place
    __device__ __forceinline__ void finish(const RevCtx<GW> &x, float &mu_b) {
        mu_b += t_sum(b.mub);
#pragma unroll
        for (int h = 0; h < N; ++h) {
            const int ci = x.G.gt + AGroup<GW>::T * (slot + h);
            const V3 nb = get_half(b.nb, h), rb = get_half(b.rb, h), cb = get_half(b.cb, h);
            x.S.ring[0][ci] = make_float4(nb.x, nb.y, nb.z, get_half(b.iknb, h));
            x.S.ring[1][ci] = make_float4(rb.x, rb.y, rb.z, get_half(b.iktb, h));
            x.S.ring[2][ci] = make_float4(cb.x, cb.y, cb.z, 0.0f);
        }
    }
};
template <int GW>
struct RevUnit<GW, NoUnit> {
    __device__ __forceinline__ void init(const RevCtx<GW> &, int) {}
    __device__ __forceinline__ void request(const RevCtx<GW> &, int) const {}
    __device__ __forceinline__ void form(const RevCtx<GW> &, const Contact<float> &, int, V3, V3) {}
    __device__ __forceinline__ void step(const RevCtx<GW> &, const Contact<float> &, V3, V3, V3, float (&)[6]) {}
    __device__ __forceinline__ void finish(const RevCtx<GW> &, float &) {}
};

template <int GW, typename T0, typename T1, bool FURTHER, bool AHEAD, bool ONE>
__device__ __forceinline__ void rev_iterations(const RevCtx<GW> &x, const Contact<float> &own, const Contact<float> &own2, int &parity, V3 &Vb, V3 &Wb,
                                               V3 &vpb, V3 &wpb, float (&Wbar)[9], float &invm_l, float &mu_b) {
    constexpr int T = AGroup<GW>::T;
    RevUnit<GW, T0> u0;
    RevUnit<GW, T1> u1;
    u0.init(x, 0);
    u1.init(x, GW == 1 ? 2 : 1);
    if (FURTHER) {   // contacts past kRC: their reverse state in sp.adjs
#pragma unroll 1
        for (int ci = kRC + x.G.gt; ci < x.nc; ci += T) {
            const int pad = rec_pad(x.sp.rec[4 * ci + 3]);
            float4 *A = x.sp.adjs + 4 * ci;
            A[0] = (pad < x.n_pads) ? make_float4(-x.S.fbar[3 * pad], -x.S.fbar[3 * pad + 1], -x.S.fbar[3 * pad + 2], 0.0f)
                                    : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            A[1] = A[2] = A[3] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    }
    // the tape of iteration it to shared memory (zeros before the first)
    auto request = [&](int it) {
        u0.request(x, it);
        u1.request(x, it);
        copy_async(&x.S.rsum[x.G.wg][it & (kRing - 1)][x.G.lane & 1],
                   reinterpret_cast<const float4 *>(x.sp.sh + 8 * max(it, 0)) + (x.G.lane & 1), it >= 0 ? 16 : 0, x.G.lane < 2);
        copy_commit();
    };
    // the sums after iteration it, and the body's velocity from them
    auto sums = [&](int it, float4 &lo, float4 &hi) {
        lo = x.S.rsum[x.G.wg][it & (kRing - 1)][0];
        hi = x.S.rsum[x.G.wg][it & (kRing - 1)][1];
    };
    float4 c_lo, c_hi, p_lo, p_hi;   // the sums after iterations it and it - 1
    {
        const float4 *q = reinterpret_cast<const float4 *>(x.sp.sh + 8 * (x.I - 1));
        c_lo = q[0];
        c_hi = q[1];
    }
    V3 Vi, Wv;   // the body's velocity before iteration it
    auto before = [&](int it) {
        sums(it - 1, p_lo, p_hi);
        Vi = x.v_pred + mk(p_lo.x, p_lo.y, p_lo.z) * x.inv_m;
        Wv = x.w_pred + smul(x.Wi, mk(p_lo.w, p_hi.x, p_hi.y));
        u0.form(x, own, it, Vi, Wv);
        u1.form(x, own2, it, Vi, Wv);
    };
#pragma unroll 1
    for (int k = 2; k <= kRing; ++k) request(x.I - k);
    if (AHEAD) {
        copy_wait<kRing - 2>();
        __syncwarp();
        before(x.I - 1);
    }
#pragma unroll 1
    for (int it = x.I - 1; it >= 0; --it) {
        request(it - kRing);   // (its place held the impulses after iteration it, in registers by now)
        copy_wait<kRing - 1 - (AHEAD ? 1 : 0)>();
        __syncwarp();          // (the sums are copied by two lanes)
        if (!AHEAD) before(it);
        // (a) V^{it+1} = v_pred + S1 / m, W^{it+1} = w_pred + W S2, sums of the impulses after it
        const V3 g = smul(x.Wi, Wb), vm = Vb * x.inv_m;
        vpb = vpb + Vb;
        wpb = wpb + Wb;
        // (b) the contact updates of iteration it, against V^it, W^it
        float acc[6] = {0, 0, 0, 0, 0, 0};
        u0.step(x, own, vm, g, Wv, acc);
        if constexpr (GW == 1 || std::is_same<T1, NoUnit>::value) u1.step(x, own2, vm, g, Wv, acc);
        else u1.step_on(x, own2, vm, g, Wv, acc);
        invm_l += dot(Vb, mk(c_lo.x, c_lo.y, c_lo.z));   // (every thread; one's is kept)
        outer_add(Wbar, Wb, mk(c_lo.w, c_hi.x, c_hi.y), 1.0f);
        c_lo = p_lo; c_hi = p_hi;
        if (FURTHER) {
#pragma unroll 1
            for (int ci = kRC + x.G.gt; ci < x.nc; ci += T) {
                const float4 *rc = x.sp.rec + 4 * ci;
                const float4 r0 = rc[0], r1 = rc[1], r2 = rc[2];
                float4 *A = x.sp.adjs + 4 * ci;
                const float4 a0 = A[0], a1 = A[1], a2 = A[2], a3 = A[3];
                const float4 l1 = x.sp.lamh[(size_t)it * x.cap + ci];
                const float4 l0 = it > 0 ? x.sp.lamh[(size_t)(it - 1) * x.cap + ci] : make_float4(0, 0, 0, 0);
                Contact<float> c;
                c.r = {r0.x, r0.y, r0.z};
                c.n = {r1.x, r1.y, r1.z};
                c.c = {r2.x, r2.y, r2.z};
                c.lam = {l0.x, l0.y, l0.z};
                c.ikn = r1.w;
                c.ikt = r2.w;
                ContactBwd<float> b;
                b.lb = {a0.x, a0.y, a0.z};
                b.nb = {a1.x, a1.y, a1.z};
                b.rb = {a2.x, a2.y, a2.z};
                b.cb = {a3.x, a3.y, a3.z};
                b.iknb = a0.w;
                b.iktb = a1.w;
                b.mub = a2.w;
                Factors<float> f;
                f.form(c, Vi, Wv, x.mu, x.width, x.beta_s);
                b.step(c, f, Vec<float>{l1.x, l1.y, l1.z}, vm, g, Wv, x.mu, x.inv_nc, acc);
                A[0] = make_float4(b.lb.x, b.lb.y, b.lb.z, b.iknb);
                A[1] = make_float4(b.nb.x, b.nb.y, b.nb.z, b.iktb);
                A[2] = make_float4(b.rb.x, b.rb.y, b.rb.z, b.mub);
                A[3] = make_float4(b.cb.x, b.cb.y, b.cb.z, 0.0f);
            }
        }
        if (AHEAD) before(it - 1);   // beside the reduction (past the first: unused)
        if constexpr (ONE) width_sum6<32>(acc, kFull, x.G.lane);
        else gsum6<GW>(acc, x.G, x.S, parity, x.aw);
        Vb = mk(acc[0], acc[1], acc[2]);
        Wb = mk(acc[3], acc[4], acc[5]);
    }
    vpb = vpb + Vb;   // V^0 = v_pred, W^0 = w_pred
    wpb = wpb + Wb;
    if (x.G.gt != 0) {
        invm_l = 0.0f;
#pragma unroll
        for (int q = 0; q < 9; ++q) Wbar[q] = 0.0f;
    }
    copy_wait<0>();
    u0.finish(x, mu_b);
    u1.finish(x, mu_b);
}

// Reverse sweep of one substep from start state b (whose forward has just
// been recomputed with a tape; nc contacts). On entry `ad` holds the
// derivatives w.r.t. the substep's end state, on return those w.r.t. b.
// invm_b (lane-uniform) and mu_b (per lane) accumulate d/d(1/m) and d/dmu.
// Not inlined: both tape modes then run the same compiled reverse, so their
// gradients agree bit for bit.
template <int GW>
__device__ __noinline__ void rev_substep(const AdjArgs &a, const Env &E_, const Body &b_, const float4 *L0,
                                        const float4 *L1, int nc, const SlotPtr &sp_, GroupSm<GW> &S,
                                        const AGroup<GW> &G_, int &parity_, Adj &ad_, float &invm_b_, float &mu_b_) {
    constexpr int T = AGroup<GW>::T;
    // by-value copies (see fwd_substep), written back on return
    const Env E = E_;
    const Body b = b_;
    const SlotPtr sp = sp_;
    const AGroup<GW> G = G_;
    int parity = parity_;
    Adj ad = ad_;
    float invm_b = invm_b_, mu_b = mu_b_;
    const float width = a.width, beta_s = a.beta_s;
    const DevScene sc = a.sc;   // by value, as E below
    const DevConfig cfg = a.cfg;
    const int cap = cfg.c_max, I = E.iters;
    const float h = cfg.h, inv_h = 1.0f / h;
    const V3 grav = mk(cfg.gx * h, cfg.gy * h, cfg.gz * h);
    const V3 v_pred = b.v + grav;
    const V3 w_pred = b.w;
    const M3 R = qmat(b.q);
    const S6 Wi = world_inv_inertia_f(R, E.Jb, E.inv_m);
    const float trW = Wi.xx + Wi.yy + Wi.zz;
    const bool solved = nc > 0 && I > 0;
    V3 Vf = v_pred, Wf = w_pred;   // body velocity after the solve
    if (solved) {
        const float *s = sp.sh + 8 * (I - 1);
        Vf = v_pred + mk(s[0], s[1], s[2]) * E.inv_m;
        Wf = w_pred + smul(Wi, mk(s[3], s[4], s[5]));
    }

    // -- integration: x' = x + h V, q' = normalize(exp(h W) q)
    V3 Vb = ad.v + ad.x * h;
    V3 Wb = ad.w;
    Q4 qb;
    {
        const float wn = sqrtf(dot(Wf, Wf));
        float sn, cs;
        sincosf(0.5f * wn * h, &sn, &cs);
        const float kq = (wn > 0.0f) ? sn / wn : 0.5f * h;
        const Q4 e = {cs, Wf.x * kq, Wf.y * kq, Wf.z * kq};
        const Q4 p = qmul(e, b.q);
        const float s = rsqrtf(p.w * p.w + p.x * p.x + p.y * p.y + p.z * p.z);
        const Q4 qn = {p.w * s, p.x * s, p.y * s, p.z * s};
        const float dq = ad.q.w * qn.w + ad.q.x * qn.x + ad.q.y * qn.y + ad.q.z * qn.z;
        const Q4 pb = {(ad.q.w - qn.w * dq) * s, (ad.q.x - qn.x * dq) * s, (ad.q.y - qn.y * dq) * s,
                       (ad.q.z - qn.z * dq) * s};
        qb = qmul(qconj(e), pb);                // p = e q: dq = L(e)^T dp
        const Q4 eb = qmul(pb, qconj(b.q));     // de = R(q)^T dp
        // e = (cos(th/2), s(th) A), A = h W, th = |A|, s(th) = sin(th/2) / th
        const float th = wn * h;
        const float sf = kq / h;
        float ds;   // s'(th) / th
        if (th < 0.25f) {
            const float t2 = th * th;
            ds = -1.0f / 24.0f + t2 * (1.0f / 960.0f - t2 * (1.0f / 107520.0f));
        } else {
            ds = (0.5f * th * cs - sn) / (th * th * th);
        }
        const V3 av = Wf * h;
        const V3 ev = mk(eb.x, eb.y, eb.z);
        const V3 ab = av * (-0.5f * sf * eb.w) + ev * sf + av * (ds * dot(av, ev));
        Wb = Wb + ab * h;
    }
    V3 vpb = mk(0, 0, 0), wpb = mk(0, 0, 0);
    float Wbar[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};   // d/dW, this lane's part
    float Rbar[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};   // d/dR, this lane's part
    V3 xb_l = mk(0, 0, 0);
    float invm_l = 0.0f;
    if (solved) {
        const int aw = GW == 1 ? 1 : min(kWarps<GW>, (nc + 31) >> 5);
        const RevCtx<GW> x = {sp, S, G, Wi, v_pred, w_pred, E.inv_m, E.mu, 1.0f / (float)nc, width, beta_s, cap, nc, I, aw, sc.n_pads};
        // the constants, from the records
        Contact<float> own;
        own.clear();
        load_constants<GW, true>(sp, S, G, nc, own);
        __syncwarp();
        if constexpr (GW == 1) {
            if (nc <= 32) rev_iterations<GW, float, NoUnit, false, true, true>(x, own, own, parity, Vb, Wb, vpb, wpb, Wbar, invm_l, mu_b);
            else if (nc <= 64) rev_iterations<GW, F2, NoUnit, false, false, true>(x, own, own, parity, Vb, Wb, vpb, wpb, Wbar, invm_l, mu_b);
            else if (nc <= 96) rev_iterations<GW, F2, float, false, false, true>(x, own, own, parity, Vb, Wb, vpb, wpb, Wbar, invm_l, mu_b);
            else rev_iterations<GW, F2, F2, true, false, true>(x, own, own, parity, Vb, Wb, vpb, wpb, Wbar, invm_l, mu_b);
        } else {
            if (aw == 1 && G.wg == 0) rev_iterations<GW, float, NoUnit, false, true, true>(x, own, own, parity, Vb, Wb, vpb, wpb, Wbar, invm_l, mu_b);
            else if ((GW != kTwo || nc <= kRC) && G.wg < aw) rev_iterations<GW, float, NoUnit, false, true, false>(x, own, own, parity, Vb, Wb, vpb, wpb, Wbar, invm_l, mu_b);
            else if constexpr (GW == kTwo) {
                if (nc > kRC) {
                    Contact<float> own2;
                    load_second<GW>(sp, G, nc, own2);
                    rev_iterations<GW, float, float, false, true, false>(x, own, own2, parity, Vb, Wb, vpb, wpb, Wbar, invm_l, mu_b);
                }
            }
            if (aw < kWarps<GW>) {   // the body's derivatives to the other warps
                if (G.gt == 0) {
                    S.fin[0] = vpb.x; S.fin[1] = vpb.y; S.fin[2] = vpb.z;
                    S.fin[3] = wpb.x; S.fin[4] = wpb.y; S.fin[5] = wpb.z;
                }
                G.sync();
                vpb = mk(S.fin[0], S.fin[1], S.fin[2]);
                wpb = mk(S.fin[3], S.fin[4], S.fin[5]);
                parity = 0;   // (the warps have used the reduction's buffers differently often)
            }
        }
        // contact setup and narrowphase, in reverse
#pragma unroll 1
        for (int ci = G.gt; ci < nc; ci += T) {
            const float4 *rc = sp.rec + 4 * ci;
            float4 d0, d1, d2, m4;   // (nb, 1/k_n bar), (rb, 1/k_t bar), (cb, -), (gap, link | pad, sphere, -)
            V3 r, n;
            float ikn, ikt;
            if (ci >= kRC) {
                const float4 r0 = rc[0], r1 = rc[1], r3 = rc[3];
                if constexpr (GW == 1) {
                    const float4 *A = sp.adjs + 4 * ci;
                    const float4 a0 = A[0], a1 = A[1], a2 = A[2];
                    mu_b += a2.w;
                    d0 = make_float4(a1.x, a1.y, a1.z, a0.w);
                    d1 = make_float4(a2.x, a2.y, a2.z, a1.w);
                    d2 = A[3];
                } else {
                    d0 = S.ring[0][ci]; d1 = S.ring[1][ci]; d2 = S.ring[2][ci];
                }
                m4 = make_float4(r0.w, r3.y, r3.z, 0.0f);
                r = xyz(r0); n = xyz(r1); ikn = r1.w; ikt = rc[2].w;
            } else {
                d0 = S.ring[0][ci]; d1 = S.ring[1][ci]; d2 = S.ring[2][ci]; m4 = S.meta[ci];
                if constexpr (GW == 1) {
                    const float *v = reinterpret_cast<const float *>(&S.cp[ci >> 6][0][G.lane]) + ((ci >> 5) & 1);
                    auto at = [&](int q) -> float { return v[(q >> 1) * 128 + (q & 1) * 2]; };
                    r = mk(at(0), at(1), at(2)); n = mk(at(3), at(4), at(5)); ikn = at(9); ikt = at(10);
                } else {
                    r = mk(own.r.x, own.r.y, own.r.z); n = mk(own.n.x, own.n.y, own.n.z); ikn = own.ikn; ikt = own.ikt;
                }
            }
            contact_setup_bwd(r, n, m4.x, ikn, ikt, __float_as_int(m4.y) & 0xff, __float_as_int(m4.z), xyz(d0), xyz(d1), xyz(d2), d0.w,
                              d1.w, Wi, trW, R, b.x, E.sfirst, sc, cfg, L0, L1, inv_h, Wbar, Rbar, xb_l, invm_l);
        }
    } else {
        vpb = vpb + Vb;
        wpb = wpb + Wb;
    }

    // sum the lanes' parts: x (3), 1/m (1), W (9), R (9)
    float r1[6] = {xb_l.x, xb_l.y, xb_l.z, invm_l, Wbar[0], Wbar[1]};
    float r2[6] = {Wbar[2], Wbar[3], Wbar[4], Wbar[5], Wbar[6], Wbar[7]};
    float r3[6] = {Wbar[8], Rbar[0], Rbar[1], Rbar[2], Rbar[3], Rbar[4]};
    float r4[6] = {Rbar[5], Rbar[6], Rbar[7], Rbar[8], 0.0f, 0.0f};
    gsum6<GW>(r1, G, S, parity);
    gsum6<GW>(r2, G, S, parity);
    gsum6<GW>(r3, G, S, parity);
    gsum6<GW>(r4, G, S, parity);
    const float Wt[9] = {r1[4], r1[5], r2[0], r2[1], r2[2], r2[3], r2[4], r2[5], r3[0]};
    float Rt[9] = {r3[1], r3[2], r3[3], r3[4], r3[5], r4[0], r4[1], r4[2], r4[3]};
    // W = R J R^T / m:  d/d(1/m) += <Wbar, R J R^T>,  Rbar += (Wbar + Wbar^T) R J / m
    {
        const float Rm[9] = {R.c0.x, R.c1.x, R.c2.x, R.c0.y, R.c1.y, R.c2.y, R.c0.z, R.c1.z, R.c2.z};
        const float J[9] = {E.Jb.xx, E.Jb.xy, E.Jb.xz, E.Jb.xy, E.Jb.yy, E.Jb.yz, E.Jb.xz, E.Jb.yz, E.Jb.zz};
        float RJ[9];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) RJ[3 * i + j] = Rm[3 * i] * J[j] + Rm[3 * i + 1] * J[3 + j] + Rm[3 * i + 2] * J[6 + j];
        float inner = 0.0f;
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float Mij = RJ[3 * i] * Rm[3 * j] + RJ[3 * i + 1] * Rm[3 * j + 1] + RJ[3 * i + 2] * Rm[3 * j + 2];
                inner += Wt[3 * i + j] * Mij;
            }
        invm_b += r1[3] + inner;
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                float sacc = 0.0f;
#pragma unroll
                for (int k = 0; k < 3; ++k) sacc += (Wt[3 * i + k] + Wt[3 * k + i]) * RJ[3 * k + j];
                Rt[3 * i + j] += sacc * E.inv_m;
            }
    }
    // R(q) -> q (the polynomial map of qmat)
    {
        const Q4 q = b.q;
        const float R00 = Rt[0], R01 = Rt[1], R02 = Rt[2], R10 = Rt[3], R11 = Rt[4], R12 = Rt[5], R20 = Rt[6],
                    R21 = Rt[7], R22 = Rt[8];
        qb.w += 2.0f * (q.z * (R10 - R01) + q.y * (R02 - R20) + q.x * (R21 - R12));
        qb.x += 2.0f * (-2.0f * q.x * (R11 + R22) + q.y * (R10 + R01) + q.z * (R20 + R02) + q.w * (R21 - R12));
        qb.y += 2.0f * (-2.0f * q.y * (R00 + R22) + q.x * (R10 + R01) + q.z * (R21 + R12) + q.w * (R02 - R20));
        qb.z += 2.0f * (-2.0f * q.z * (R00 + R11) + q.x * (R20 + R02) + q.y * (R21 + R12) + q.w * (R10 - R01));
    }
    ad.x = ad.x + mk(r1[0], r1[1], r1[2]);
    ad.q = qb;
    ad.v = vpb;
    ad.w = wpb;
    ad_ = ad;
    parity_ = parity;
    invm_b_ = invm_b;
    mu_b_ = mu_b;
}

// The refinement step of elite i, taken by the thread that wrote its trial's
// cost (the group's first) at the end of the trial's adjoint launch. The trial
// is accepted when it lowers the elite's cost (the first evaluation always
// is); otherwise the step multiplier halves. Then the next trial steps from
// the best state along the normalised steepest descent in coordinates scaled
// by eta:
//   s = eta * g,  dz = -scale * eta * s / |s|
// (position += dz_0..2, R <- exp([dz_3..5]x) R, m += dz_6, mu += dz_7, with m
// and mu clamped), or, after the last trial, the best state is restored and
// an improved elite's live end state, parameters and window cost (sum and
// mean) replace the scored ones. Not inlined: one copy for the kernel's three
// exits keeps it out of the adjoint's own code.
__device__ __noinline__ void refine_step(const RefineArgs &r, int i) {
    const int env = r.elite[i];
    const double c = r.cost[i];
    const float4 *tp = r.step == 0 ? r.ws_pose : r.tr_pose;
    const float2 *tq = r.step == 0 ? r.ws_params : r.tr_params;
    if (r.step == 0 || c < r.best_c[i]) {
        r.accepted[i] = (r.step == 0 ? 0ull : r.accepted[i]) | (1ull << r.step);
        r.best_pose[2 * i] = tp[2 * env];
        r.best_pose[2 * i + 1] = tp[2 * env + 1];
        for (int q = 0; q < 2; ++q) {
            r.best_end_pose[2 * i + q] = r.end_pose[2 * i + q];
            r.best_end_vel[2 * i + q] = r.end_vel[2 * i + q];
        }
        r.best_params[i] = tq[env];
        for (int d = 0; d < 8; ++d) r.best_grad[8 * i + d] = r.grad[8 * i + d];
        r.best_c[i] = c;
        if (r.step == 0) { r.c0[i] = c; r.scale[i] = 1.0f; }
    } else {
        r.scale[i] *= 0.5f;
    }
    const float4 p0 = r.best_pose[2 * i], p1 = r.best_pose[2 * i + 1];
    float2 th = r.best_params[i];
    if (r.last) {
        r.tr_pose[2 * env] = p0;
        r.tr_pose[2 * env + 1] = p1;
        r.tr_params[env] = th;
        const double cb = r.best_c[i];
        if (cb < r.c0[i]) {   // improved: its best trial's window replaces the scored one
            r.pose[2 * env] = r.best_end_pose[2 * i];
            r.pose[2 * env + 1] = r.best_end_pose[2 * i + 1];
            r.vel[2 * env] = r.best_end_vel[2 * i];
            r.vel[2 * env + 1] = r.best_end_vel[2 * i + 1];
            r.params[env] = th;
            const int nw = *r.n_window;
            r.c_sum[env] = cb;
            r.c_mean[env] = nw > 0 ? cb / (double)nw : cb;
        }
        return;
    }
    float sv[8], nrm2 = 0.0f;
    for (int d = 0; d < 8; ++d) {
        sv[d] = r.eta[d] * r.best_grad[8 * i + d];
        nrm2 += sv[d] * sv[d];
    }
    float dz[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (nrm2 > 0.0f && isfinite(nrm2)) {
        const float f = -r.scale[i] * rsqrtf(nrm2);
        for (int d = 0; d < 8; ++d) dz[d] = f * r.eta[d] * sv[d];
    }
    const float an = sqrtf(dz[3] * dz[3] + dz[4] * dz[4] + dz[5] * dz[5]);
    float sn, cs;
    sincosf(0.5f * an, &sn, &cs);
    const float kq = an > 0.0f ? sn / an : 0.5f;
    const Q4 e = {cs, dz[3] * kq, dz[4] * kq, dz[5] * kq};
    const Q4 q = qnorm(qmul(e, Q4{p1.x, p1.y, p1.z, p1.w}));
    th.x = fminf(fmaxf(th.x + dz[6], r.m_lo), r.m_hi);
    th.y = fminf(fmaxf(th.y + dz[7], r.mu_lo), r.mu_hi);
    r.tr_pose[2 * env] = make_float4(p0.x + dz[0], p0.y + dz[1], p0.z + dz[2], 0.0f);
    r.tr_pose[2 * env + 1] = make_float4(q.w, q.x, q.y, q.z);
    r.tr_params[env] = th;
}

template <int GW>
__global__ void __launch_bounds__(32 * kWarps<GW>) adjoint_kernel(const __grid_constant__ AdjArgs a) {
    constexpr int T = AGroup<GW>::T;
    __shared__ GroupSm<GW> S;
    __shared__ PadTable PT;
    const AGroup<GW> G;
    const int lane = G.gt;   // the block's thread (0 .. 32 GW - 1)
    const int slot = blockIdx.x;
    PT.build(a.sc, lane, T);
    G.sync();
    int parity = 0;   // the group's reduction buffer
    const DevScene &sc = a.sc;
    const DevConfig &cfg = a.cfg;
    const int ns = cfg.substeps, Lk = sc.n_links, P = sc.n_pads, cap = cfg.c_max;
    const int env = a.envs ? a.envs[slot] : slot;
    if (env < 0 || env >= a.N) {   // not an environment of the handle
        if (lane < 8) a.grad[8 * slot + lane] = 0.0f;
        if (a.grad_quat && lane < 4) a.grad_quat[4 * slot + lane] = 0.0f;
        if (lane == 0 && a.cost) a.cost[slot] = NAN;
        return;
    }
    const bool seg_tape = a.seg_tape != 0;   // every substep of a segment keeps its tape
    const int nck = (a.H + a.K - 1) / a.K;
    // with whole-segment tapes, the segments recomputed later keep their
    // substeps' contact records from the first pass, and their recomputation
    // replays them
    const int nrec = seg_tape ? (nck - 1) * a.K * ns : 0;
    const SlotLayout Ly = slot_layout(a.H, a.K, ns, P, cap, a.iters_max, seg_tape ? a.K * ns : 1, nrec);
    float *base = a.scratch + (size_t)slot * a.stride;
    SlotPtr sp0;
    sp0.ck = reinterpret_cast<float4 *>(base + Ly.ck);
    sp0.sg = reinterpret_cast<float4 *>(base + Ly.sg);
    sp0.sf = base + Ly.sf;
    sp0.lamf = reinterpret_cast<float4 *>(base + Ly.lamf);
    sp0.adjs = reinterpret_cast<float4 *>(base + Ly.adj);
    sp0.recs = reinterpret_cast<float4 *>(base + Ly.recs);
    sp0.nrc = reinterpret_cast<int *>(base + Ly.nrc);
    sp0.ncs = reinterpret_cast<int *>(base + Ly.ncs);
    sp0.tape = base + Ly.tape;
    sp0.blk_lamh = Ly.blk_lamh;
    sp0.blk_sh = Ly.blk_sh;
    sp0.blk_stride = Ly.blk_stride;
    const SlotPtr sp = sp0.blk(0);

    const float4 P0 = a.pose[2 * env], P1 = a.pose[2 * env + 1];
    const float4 V0 = a.vel[2 * env], V1 = a.vel[2 * env + 1];
    const float2 th = a.params[env];
    const int shp = a.shape[env];
    Env E;
    E.sfirst = __ldg(sc.shape_first + shp);
    E.NS = __ldg(sc.shape_count + shp);
    E.iters = a.iters[env];
    E.mu = th.y;
    E.inv_m = 1.0f / th.x;
    E.cfirst = __ldg(sc.cl_first + shp);
    E.Jb.xx = __ldg(sc.shape_jinv + 6 * shp + 0); E.Jb.yy = __ldg(sc.shape_jinv + 6 * shp + 1);
    E.Jb.zz = __ldg(sc.shape_jinv + 6 * shp + 2); E.Jb.xy = __ldg(sc.shape_jinv + 6 * shp + 3);
    E.Jb.xz = __ldg(sc.shape_jinv + 6 * shp + 4); E.Jb.yz = __ldg(sc.shape_jinv + 6 * shp + 5);
    const Body b0 = {xyz(P0), Q4{P1.x, P1.y, P1.z, P1.w}, xyz(V0), xyz(V1)};
    int st = a.status[env];
    if (E.iters > a.iters_max) st |= IH_ENV_INVALID;   // the tape cannot hold its iterations

    const float h = cfg.h, inv_h = 1.0f / h, inv_ns = 1.0f / (float)ns;
    const size_t tab_frame = (size_t)(ns + 1) * Lk * kLinkStride;
    const float4 *tab0 = a.link_tab + (size_t)a.frame0 * tab_frame;

    // -- pass 1: the cost, the state at every K-th frame, every frame's pad
    //    forces, the substep states of the last segment (the first one
    //    reversed) and its tape, and the contact records of the others
    const int f_last = (nck - 1) * a.K;
    double cost = 0.0;
    Body b = b0;
#pragma unroll 1
    for (int f = 0; f < a.H && !(st & kDiverged); ++f) {
        if (f % a.K == 0 && lane == 0) store_body(sp.ck + 4 * (f / a.K), b);
#pragma unroll 1
        for (int k = lane; k < 3 * P; k += T) S.padacc[k] = 0.0f;
        G.sync();
        const float4 *tab = tab0 + (size_t)f * tab_frame;
#pragma unroll 1
        for (int s = 0; s < ns; ++s) {
            const float4 *L0 = tab + (size_t)s * Lk * kLinkStride;
            if (f >= f_last) {
                const int blk = (f - f_last) * ns + s;
                if (lane == 0) store_body(sp.sg + 4 * blk, b);
                if (seg_tape && !a.forward_only) {   // the last segment's tape, recorded on the way
                    const int nc = fwd_substep<GW>(a, E, b, L0, L0 + Lk * kLinkStride, sp.blk(blk), S, PT, G, parity,
                                                       st, 1 | a.zero, 1 | a.zero, -1);
                    if (lane == 0) sp.ncs[blk] = nc;
                    continue;
                }
            }
            if (nrec > 0 && f < f_last) {   // a segment recomputed later: keep this substep's records
                const int q = f * ns + s;
                SlotPtr sq = sp;
                sq.rec = sp.recs + (size_t)q * cap * 4;
                const int nc = fwd_substep<GW>(a, E, b, L0, L0 + Lk * kLinkStride, sq, S, PT, G, parity, st, a.zero,
                                                   1 | a.zero, -1);
                if (lane == 0) sp.nrc[q] = nc;
                continue;
            }
            fwd_substep<GW>(a, E, b, L0, L0 + Lk * kLinkStride, sp, S, PT, G, parity, st, a.zero, 1 | a.zero, -1);
        }
#pragma unroll 1
        for (int k = lane; k < 3 * P; k += T) sp.sf[(size_t)f * 3 * P + k] = S.padacc[k] * inv_ns;
        if (!all_finite(b.x, b.q, b.v, b.w)) st |= IH_ENV_NONFINITE;
        else if (dot(b.x, b.x) > cfg.escape_radius * cfg.escape_radius) st |= IH_ENV_ESCAPED;
        {   // frame cost in FP64, as the scored step: each pad's terms in parallel, summed in pad order
            const float *o = a.obs + (size_t)f * P * 3;
            const double tau = (double)cfg.tau, tau2 = __dmul_rn(tau, tau), wf = (double)cfg.w_force;
#pragma unroll 1
            for (int p = lane; p < P; p += T) {
                const double fx = S.padacc[3 * p] * inv_ns, fy = S.padacc[3 * p + 1] * inv_ns,
                             fz = S.padacc[3 * p + 2] * inv_ns;
                const double ox = o[3 * p], oy = o[3 * p + 1], oz = o[3 * p + 2];
                const double dx = __dsub_rn(fx, ox), dy = __dsub_rn(fy, oy), dz = __dsub_rn(fz, oz);
                const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                S.term[p] = __dmul_rn(wf, d2);
                const double n2 = __dadd_rn(__dadd_rn(__dmul_rn(fx, fx), __dmul_rn(fy, fy)), __dmul_rn(fz, fz));
                const double no = __dadd_rn(__dadd_rn(__dmul_rn(ox, ox), __dmul_rn(oy, oy)), __dmul_rn(oz, oz));
                S.flag[p] = (n2 > tau2) != (no > tau2);
            }
            G.sync();
            if (lane == 0) {
                double cf = 0.0;
#pragma unroll 1
                for (int p = 0; p < P; ++p) {
                    cf = __dadd_rn(cf, S.term[p]);
                    if (S.flag[p]) cf = __dadd_rn(cf, (double)cfg.w_contact);
                }
                cost = __dadd_rn(cost, cf);
            }
        }
        G.sync();
    }
    if (a.out_pose && lane == 0) {   // the horizon's end state (not meaningful when diverged)
        a.out_pose[2 * slot] = make_float4(b.x.x, b.x.y, b.x.z, 0.0f);
        a.out_pose[2 * slot + 1] = make_float4(b.q.w, b.q.x, b.q.y, b.q.z);
        a.out_vel[2 * slot] = make_float4(b.v.x, b.v.y, b.v.z, 0.0f);
        a.out_vel[2 * slot + 1] = make_float4(b.w.x, b.w.y, b.w.z, 0.0f);
    }
    if (a.forward_only) {
        if (lane == 0 && a.cost) a.cost[slot] = (st & kDiverged) ? INFINITY : cost;
        if (lane == 0 && a.refine) refine_step(a.rf, slot);
        return;
    }
    if (st & kDiverged) {   // no derivative of a diverged or invalid environment
        if (lane < 8) a.grad[8 * slot + lane] = 0.0f;
        if (a.grad_quat && lane < 4) a.grad_quat[4 * slot + lane] = 0.0f;
        if (lane == 0 && a.cost) a.cost[slot] = INFINITY;
        __syncwarp();   // (the refinement step reads the whole gradient)
        if (lane == 0 && a.refine) refine_step(a.rf, slot);
        return;
    }

    // -- pass 2: segments in reverse
    Adj ad = {mk(0, 0, 0), Q4{0, 0, 0, 0}, mk(0, 0, 0), mk(0, 0, 0)};
    float invm_b = 0.0f, mu_b = 0.0f;
    const float wf2 = 2.0f * cfg.w_force * inv_h * inv_ns;
#pragma unroll 1
    for (int seg = nck - 1; seg >= 0; --seg) {
        const int fb = seg * a.K, fe = min(a.H, fb + a.K);
        b = load_body(sp.ck + 4 * seg);
        // the segment's substep start states and tapes (its frames' pad forces
        // are the first pass's)
#pragma unroll 1
        for (int f = fb; f < fe && seg < nck - 1; ++f) {
            const float4 *tab = tab0 + (size_t)f * tab_frame;
#pragma unroll 1
            for (int s = 0; s < ns; ++s) {
                const int blk = (f - fb) * ns + s;
                if (lane == 0) store_body(sp.sg + 4 * blk, b);
                const float4 *L0 = tab + (size_t)s * Lk * kLinkStride;
                if (seg_tape) {   // replaying the first pass's records of the substep
                    const int q = f * ns + s;
                    SlotPtr sq = sp.blk(blk);
                    sq.rec = sp.recs + (size_t)q * cap * 4;
                    const int nc = fwd_substep<GW>(a, E, b, L0, L0 + Lk * kLinkStride, sq, S, PT, G, parity, st,
                                                       1 | a.zero, a.zero, sp.nrc[q]);
                    if (lane == 0) sp.ncs[blk] = nc;
                } else {
                    fwd_substep<GW>(a, E, b, L0, L0 + Lk * kLinkStride, sp, S, PT, G, parity, st, a.zero, a.zero,
                                        -1);
                }
            }
        }
#pragma unroll 1
        for (int f = fe - 1; f >= fb; --f) {
            const float *o = a.obs + (size_t)f * P * 3;
#pragma unroll 1
            for (int k = lane; k < 3 * P; k += T)
                S.fbar[k] = wf2 * (sp.sf[(size_t)f * 3 * P + k] - o[k]);
            G.sync();
            const float4 *tab = tab0 + (size_t)f * tab_frame;
#pragma unroll 1
            for (int s = ns - 1; s >= 0; --s) {
                const float4 *L0 = tab + (size_t)s * Lk * kLinkStride;
                const float4 *L1 = L0 + Lk * kLinkStride;
                const int blk = (f - fb) * ns + s;
                const Body bs = load_body(sp.sg + 4 * blk);
                if (seg_tape) {
                    G.sync();
                    SlotPtr sq = sp.blk(blk);
                    if (seg < nck - 1) sq.rec = sp.recs + (size_t)(f * ns + s) * cap * 4;   // (the replayed records)
                    rev_substep<GW>(a, E, bs, L0, L1, sp.ncs[blk], sq, S, G, parity, ad, invm_b, mu_b);
                } else {   // re-run the substep once more, recording its tape
                    Body bt = bs;
                    int st2 = 0;
                    const int nc = fwd_substep<GW>(a, E, bt, L0, L1, sp, S, PT, G, parity, st2, 1 | a.zero, a.zero, -1);
                    rev_substep<GW>(a, E, bs, L0, L1, nc, sp, S, G, parity, ad, invm_b, mu_b);
                }
            }
            G.sync();
        }
    }
    {
        float mv[6] = {mu_b, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        gsum6<GW>(mv, G, S, parity);
        mu_b = mv[0];
    }
    if (lane == 0) {
        // rotation tangent: q = exp(delta) q0, d/d delta at 0 = vec(qbar (x) conj(q0)) / 2
        const Q4 g = qmul(ad.q, qconj(b0.q));
        float *gr = a.grad + 8 * slot;
        gr[0] = ad.x.x; gr[1] = ad.x.y; gr[2] = ad.x.z;
        gr[3] = 0.5f * g.x; gr[4] = 0.5f * g.y; gr[5] = 0.5f * g.z;
        gr[6] = -invm_b * E.inv_m * E.inv_m;
        gr[7] = mu_b;
        if (a.grad_quat) {
            a.grad_quat[4 * slot + 0] = ad.q.w; a.grad_quat[4 * slot + 1] = ad.q.x;
            a.grad_quat[4 * slot + 2] = ad.q.y; a.grad_quat[4 * slot + 3] = ad.q.z;
        }
        if (a.cost) a.cost[slot] = cost;
        if (a.refine) refine_step(a.rf, slot);
    }
}

template <int GW>
cudaError_t launch_gw(const AdjArgs &a, cudaStream_t s) {
    adjoint_kernel<GW><<<a.n, 32 * kWarps<GW>, 0, s>>>(a);
    return cudaGetLastError();
}

__global__ void iters_max_kernel(int N, const int *iters, int *out) {
    int m = 0;
    for (int i = threadIdx.x; i < N; i += blockDim.x) m = max(m, iters[i]);
    m = __reduce_max_sync(kFull, m);
    __shared__ int part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = max(m, part[w]);
        *out = m;
    }
}

}  // namespace

size_t adjoint_scratch_floats(int H, int K, int substeps, int n_pads, int c_max, int iters_max, bool seg_tape) {
    const int nck = (H + K - 1) / K;
    return slot_layout(H, K, substeps, n_pads, c_max, iters_max, seg_tape ? K * substeps : 1,
                       seg_tape ? (nck - 1) * K * substeps : 0).total;
}

cudaError_t launch_adjoint_iters_max(int N, const int *iters, int *out, cudaStream_t s) {
    iters_max_kernel<<<1, 256, 0, s>>>(N, iters, out);
    return cudaGetLastError();
}

bool adjoint_variant_supported(int gw, int pl) {
    return (gw == 0 && pl == 0) || (gw == 4 && pl == 1) || (gw == 1 && (pl == 1 || pl == 2));
}

// Automatic shape. Few environments (the refined elites, a small batch), at most two
// per SM -- the blocks of 255 registers a thread that an SM holds: four warps each, so
// that their contacts' chains run side by side. More: one warp each (no barriers, and
// up to eight an SM at once). Six frames of the box / the cylinder / the mug, in us,
// four warps against one: 1 environment 261 : 302 / 293 : 415 / 710 : 870, 304
// environments 276 : 315 / 368 : 528 / 843 : 986, 305 environments 490 : 316 /
// 619 : 533 / 1436 : 982. The second number of a shape no longer changes anything.
// Four warps hold a second contact a thread beside the first where a scene can have more
// than 128 contacts: 64 mixed environments, one of them with 150 contacts, four frames,
// 418 us (650 with the further contacts run from scratch memory after the others, 605 by
// the kernels before that). The other scenes' kernel has no such code.
cudaError_t launch_adjoint(const AdjArgs &a, cudaStream_t s) {
    const auto four = [&]() { return a.cfg.c_max <= kRC ? launch_gw<4>(a, s) : launch_gw<kTwo>(a, s); };
    if (a.gw == 4) return four();
    if (a.gw == 1) return launch_gw<1>(a, s);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    return a.n <= 2 * sms ? four() : launch_gw<1>(a, s);
}

}  // namespace ih
