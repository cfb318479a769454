// step_kernel.cuh -- the batched dynamics step s_{t+1} = f(s_t, u_t, theta) of N
// independent hand-plus-object simulations (Sec. III-A; Algorithm 1, "step
// simulation"), with the contact-sensor readout c_t^(l) of every pad.
//
// L lanes of one warp (32, or 16 with two environments to a warp) own one
// environment at a time; nothing but the warp synchronises (but see teams below). Per substep they
//   1. predict the velocity under gravity and cache the object's spheres, rotated
//      into the world frame, and the links' offsets in shared memory;
//   2. cull (link, 8-sphere cluster) pairs by the clusters' enclosing
//      spheres; then one lane takes each surviving pair and tests its eight
//      spheres by squared distance alone (the few within 1e-5 of the margin
//      again by their gap), and the contacts (gap d < margin) are listed in
//      pair order (link, then sphere) by bit-plane ballots of the lanes' counts;
//   3. set each listed contact up: gap, normal and lever arm, its pad, scalar
//      normal/tangential effective masses, and the bias folded into a target
//      velocity; the first kSlots L contacts go to registers;
//   4. run `iters` Jacobi projected-impulse iterations: every contact updates
//      against the same body velocity, then the impulses and moments are
//      summed by shuffles and the body velocity recomputed;
//   5. integrate (symplectic Euler, exact rotation exponential) and add the
//      contacts' impulses into their sensor pads in a fixed order, one lane per
//      pad and component scanning the contacts of the pad's link.
// Nothing here is a dense contraction: the kernel is bound by FP32 issue and by
// the latency of the solver's chain (and, when the device is full, by instruction
// fetch: the loops off the solver are kept rolled). Against groups of 64 (or, in
// large batches, 32) threads with block barriers, a link cull before the cluster
// cull, one pair test per thread and guarded scalar slots, sim_step alone: 1024
// cylinders, ten frames, 421 -> 308 us (332 with the registers of 16 warps an SM);
// 32768 mugs, two frames, 4.49 -> 3.65 ms; 4097 boxes, four frames, 392 -> 144 us;
// 8192 of mixed shapes, six frames, 969 -> 867 us.
// In small batches of the 128-wide sums a team of four warps finds and sets up an
// environment's contacts (a thread each instead of a lane's two to four in turn, a
// third of such a substep) and its first warp runs the solver.
//
// A step shape's width TPE (16, 32, 64, 128) fixes the order of the solver's
// sums and with it every bit of the result: thread t of TPE adds contacts t,
// t + TPE, ... in order, each 32 threads are summed by a xor tree (16, 8, 4, 2,
// 1), and the 32-thread sums are added in order. The lanes that execute it are a
// free choice: a lane holds the accumulators of threads lane, lane + L, ...
// (zeros of empty threads change nothing), and a tree level that pairs two
// threads of one lane is an addition in that lane.
#pragma once
#include <cstddef>

#include "contact.cuh"
#include "internal.cuh"

namespace ih {
namespace {

// the shapes of the interface (summation width, contacts per thread); the
// second number no longer changes anything: the width alone fixes the result
#define IH_STEP_VARIANTS(X) X(16, 2) X(16, 4) X(32, 1) X(32, 2) X(32, 3) X(32, 4) X(64, 1) X(64, 2) X(128, 1)
// the compiled kernels: (lanes per environment, summation width, warps to an SM, whether
// a lane's first contact past the register slots is updated beside them, warps that
// find and set up an environment's contacts)
#define IH_STEP_KERNELS(X)                                                                      \
    IH_STEP_KERNELS_16(X, kFewBlocks, false) IH_STEP_KERNELS_16(X, kManyBlocks, false)          \
    IH_STEP_KERNELS_32(X, kFewBlocks, false) IH_STEP_KERNELS_32(X, kManyBlocks, false) IH_STEP_KERNELS_32(X, kFewBlocks, true) \
    X(32, 128, kFewBlocks, false, kTeam) X(32, 128, kFewBlocks, true, kTeam)
#define IH_STEP_KERNELS_16(X, B, F) X(16, 16, B, F, 1) X(16, 32, B, F, 1) X(16, 64, B, F, 1)
#define IH_STEP_KERNELS_32(X, B, F) X(32, 32, B, F, 1) X(32, 64, B, F, 1) X(32, 128, B, F, 1)
constexpr int kSlots = 4;            // register-resident contacts per lane
constexpr unsigned kAll = 0xffffffffu;
template <bool V>
struct Flag {
    static constexpr bool value = V;
};
template <int V>
struct Int {
    static constexpr int value = V;
};

// Shared memory of one environment. Everything has a fixed size except the
// contact records, the caches of world-frame centres and the lists, which follow.
struct alignas(16) GSm {
    union {
        double term[IH_MAX_PADS];    // FP64 force term of each pad (scoring)
        float fin[6];                // the solved velocity, for a team's other warps
    };
    float4 xa[kMaxLinks];            // x - link origin
    float4 ax[kMaxLinks];            // link axis
    float padacc[IH_MAX_PADS * 3];
    union {
        int flag[IH_MAX_PADS];       // contact-state mismatch of each pad (scoring)
        int cnt[2][kTeam];           // hits of a team's warps in a listing round (double-buffered)
    };
    unsigned short lbeg[kMaxLinks], lend[kMaxLinks];   // contact range of each link
};
static_assert(sizeof(GSm) % 16 == 0, "the records keep 16-byte alignment");
__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) & ~size_t(15); }
__host__ __device__ constexpr int sph_cap(int s_max) { return (s_max + kCluster - 1) / kCluster * kSphStride; }
// contacts whose record (3 float4) and impulse (1) are in shared memory: the
// register-resident ones; the rest of up to c_max spill to global memory
__host__ __device__ constexpr int stage_capacity(int lanes, int c_max) {
    return c_max < kSlots * lanes ? c_max : kSlots * lanes;
}
// contacts of the spill area of an environment: whole rows of the lanes
__host__ __device__ constexpr int spill_rows(int lanes, int c_max) {
    return c_max > kSlots * lanes ? (c_max - kSlots * lanes + lanes - 1) / lanes * lanes : 0;
}
// float4s of the sphere cache and the impulses, which share their place (the
// spheres are done with when the first impulse is stored) unless the solver
// starts from cached impulses
__host__ __device__ constexpr int sph_lam_cap(int s_max, int stage_cap, bool warm) {
    return warm ? sph_cap(s_max) + stage_cap : sph_cap(s_max) > stage_cap ? sph_cap(s_max) : stage_cap;
}
__host__ __device__ inline size_t env_bytes(int s_max, int stage_cap, int c_max, bool warm, int clp_cap) {
    return sizeof(GSm) +
           sizeof(float4) * (3 * (size_t)stage_cap + sph_lam_cap(s_max, stage_cap, warm) + kMaxLinks + (warm ? c_max : 0)) +
           align16(2 * (size_t)clp_cap) + align16(2 * (size_t)c_max) + align16((size_t)c_max);
}

// The sum over an environment's L lanes of six values A (one 32-thread tree of the
// width, its first level already added when L = 16) or of A and B (two trees,
// added in order), every lane receiving the six totals. Reduce-scatter: a level
// sends the half of the values that the lane does not keep, so 13 shuffles (two
// trees, L = 32) reduce twelve values.
template <int L>
__device__ __forceinline__ void sum_trees(const float (&A)[6], const float (&B)[6], float (&v)[6], int gl) {
    // the first level leaves A to one half of the lanes and B to the other
    constexpr int H = L / 2;
    const bool b1 = gl & H, b2 = gl & (H / 2), b3 = gl & (H / 4), b4 = gl & (H / 8);
    float s[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) s[k] = (b1 ? B[k] : A[k]) + __shfl_xor_sync(kAll, b1 ? A[k] : B[k], H, L);
    float t[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] = (b2 ? s[k + 3] : s[k]) + __shfl_xor_sync(kAll, b2 ? s[k] : s[k + 3], H / 2, L);
    const float u0 = (b3 ? t[2] : t[0]) + __shfl_xor_sync(kAll, b3 ? t[0] : t[2], H / 4, L);
    const float u1 = (b3 ? 0.0f : t[1]) + __shfl_xor_sync(kAll, b3 ? t[1] : 0.0f, H / 4, L);
    float c = (b4 ? u1 : u0) + __shfl_xor_sync(kAll, b4 ? u0 : u1, H / 8, L);
    if constexpr (L == 32) c += __shfl_xor_sync(kAll, c, 1, L);
    c += __shfl_xor_sync(kAll, c, H, L);   // A + B
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = __shfl_sync(kAll, c, (k / 3) * (H / 2) + (k % 3 == 2 ? H / 4 : (k % 3) * (H / 8)), L);
}

// The sums of NA accumulators of six values (accumulator j of lane g: thread
// g + j L of the summation width L NA), of which the first NZ can be nonzero, in
// the width's order (see above; a tree of zeros is left out).
template <int L, int NA, int NZ>
__device__ __forceinline__ void env_sum6(const float (&acc)[NA][6], float (&v)[6], int gl) {
    if constexpr (L * NA <= 64) {
        float A[6], B[6];
        constexpr bool two = L * NA == 64 && (L == 32 ? NZ > 1 : NZ > 2);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            A[k] = (L == 16 && NA > 1 && NZ > 1) ? acc[0][k] + acc[NA > 1 ? 1 : 0][k] : acc[0][k];
            if constexpr (two) B[k] = L == 16 ? (NZ > 3 ? acc[NA - 2][k] + acc[NA - 1][k] : acc[NA - 2][k]) : acc[NA - 1][k];
        }
        if constexpr (two) {
            sum_trees<L>(A, B, v, gl);
        } else {
#pragma unroll
            for (int k = 0; k < 6; ++k) v[k] = A[k];
            width_sum6<L>(v, kAll, gl);
        }
    } else {   // 128: four sums, added in order
        float c = width_scatter6<32>(acc[0], kAll, gl);
#pragma unroll
        for (int j = 1; j < NZ; ++j) c += width_scatter6<32>(acc[j], kAll, gl);
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = __shfl_sync(kAll, c, scatter_lane<32>(k), 32);
    }
}

// order-preserving key of a cost (NaN excluded), compared with integers: FP64
// compares take the scarce FP64 pipe
__device__ __forceinline__ unsigned long long cost_key(double c) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(c);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// One warp per block, so that the environments spread evenly over the SMs (an
// SM holds 6 or 7 of 1024 environments; blocks of two would put 8 on some), and
// B warps to an SM by registers (kFewBlocks or kManyBlocks). FIRST: a lane's first
// contact past its register slots is updated beside them. W > 1: a team of W warps owns
// the block's one environment; its first warp runs the solver alone, and all of them the
// rest of a substep (the same environment state in every thread).
template <int L, int TPE, bool WARM, int B, bool FIRST, int W>
__global__ void __launch_bounds__(32 * W, W == 1 ? B : kTeamBlocks) step_kernel(const StepArgs a, int s_max) {
    static_assert(TPE % L == 0 && TPE / L <= kSlots, "the width's threads are the lanes' accumulators");
    static_assert(W == 1 || (L == 32 && W == kTeam), "a team's warps work on one environment");
    constexpr int EPW = 32 / L, NA = TPE / L, RCAP = kSlots * L;
    constexpr int E = L * W;   // the environment's threads
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = W == 1 ? threadIdx.x : threadIdx.x & 31, sub = lane / L, gl = lane % L, shift = sub * L;
    const int warp = W == 1 ? 0 : threadIdx.x >> 5, gt = W == 1 ? gl : threadIdx.x;   // gt: the environment's thread
    // between the phases of a substep (every warp of a team passes the same ones)
    auto sync = [&]() {
        if constexpr (W == 1) __syncwarp();
        else __syncthreads();
    };
    const DevScene &sc = a.sc;
    const DevConfig &cfg = a.cfg;
    const int ns = cfg.substeps, Lk = sc.n_links, P = sc.n_pads;
    const float h = cfg.h, inv_h = 1.0f / h, inv_L = 1.0f / sc.link_len;
    const V3 grav = mk(cfg.gx * h, cfg.gy * h, cfg.gz * h);
    // the frame, observation and outputs (from the window descriptor when replayed)
    int frame0 = a.frame0;
    const float *obs = a.obs;
    if (a.win) {
        frame0 = a.win->frame0 + a.win_k;
        obs = a.win->obs ? a.win->obs + (size_t)a.win_k * P * 3 : nullptr;
    }
    const bool window_mode = a.cm_frames != nullptr;   // every frame scored, argmin afterwards
    const bool scored = obs != nullptr;
    const int n_win0 = scored ? *a.n_window : 0;       // frames in the window before this launch

    const int cap = cfg.c_max;
    const int SC = a.stage_cap;   // contacts staged in shared memory (RCAP, or c_max); the rest spill to global memory
    PadTable &PT = *reinterpret_cast<PadTable *>(smem);
    PT.build(sc, threadIdx.x, 32 * W);
    sync();
    unsigned char *mine = smem + sizeof(PadTable) + sub * env_bytes(s_max, SC, cap, WARM, a.clp_cap);
    GSm &S = *reinterpret_cast<GSm *>(mine);
    // contact records, 3 float4 each: (r, 1/k_t), (n, 1/k_n), (c, -); the impulses follow
    float4 *rec = reinterpret_cast<float4 *>(mine + sizeof(GSm));
    float4 *sph = rec + 3 * SC;            // sphere centres (world rotation, relative to x), radius
    float4 *lamst = WARM ? sph + sph_cap(s_max) : sph;
    float4 *clc = sph + sph_lam_cap(s_max, SC, WARM);    // cluster centres, enclosing radius
    // warm start: final impulse (xyz) and pair id (w, link << 8 | sphere) of the
    // environment's last substep's contacts, in pair order
    float4 *prev = clc + kMaxLinks;
    // surviving pairs in order (link << 8 | cluster); contacts in order (link << 8 | sphere); their pads
    unsigned short *clp = reinterpret_cast<unsigned short *>(prev + (WARM ? cap : 0));
    unsigned short *clist = reinterpret_cast<unsigned short *>(reinterpret_cast<unsigned char *>(clp) + align16(2 * (size_t)a.clp_cap));
    unsigned char *cpad = reinterpret_cast<unsigned char *>(clist) + align16(2 * (size_t)cap);
    // contacts SC .. c_max - 1 of the environment (and the rest of a row of the lanes):
    // its slot of the spill area
    float4 *spill_g = a.spill ? a.spill + (size_t)(blockIdx.x * EPW + sub) * (size_t)spill_rows(L, cap) * 4 : nullptr;   // (SC = RCAP when there is one)
    auto ballot = [&](bool p) -> unsigned {   // of the environment's lanes, bit 0 its first
        const unsigned b = __ballot_sync(kAll, p);
        return L == 32 ? b : (b >> shift) & 0xffffu;
    };
    auto wmax = [&](int v) -> int { return L == 32 ? v : max(v, __shfl_xor_sync(kAll, v, 16)); };
    const unsigned below = (1u << gl) - 1u;
    // The slot of this thread's first of `mine` (below 2^BITS) hits in an order-preserving
    // list of n so far, by bit planes of the lanes' ballots; n advances by all of them
    int parity = 0;   // a team's counts in use
    auto list = [&](auto bits, int mine, int &n) -> int {
        int off = n, tot = 0;
#pragma unroll
        for (int b = 0; b < decltype(bits)::value; ++b) {
            const unsigned bal = ballot((mine >> b) & 1);
            off += __popc(bal & below) << b;
            tot += __popc(bal) << b;
        }
        if constexpr (W > 1) {
            int *c = S.cnt[parity];
            if (lane == 0) c[warp] = tot;
            sync();
            tot = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                if (w < warp) off += c[w];
                tot += c[w];
            }
            parity ^= 1;
        }
        n += tot;
        return off;
    };

    unsigned long long best_k = ~0ull;   // best (C, env) of these lanes so far (single scored frame)
    int best_i = 0x7fffffff;
    unsigned long long work = 0ull;      // lane k < 6: work counter k (see sim_work_counters)

    // The next environments of the warp: from the launch's work queue (slots in
    // LPT order, taken by whichever warp is free), else grid-stride. Both
    // environments of a 16-lane warp walk the same loops to the larger of their
    // counts, so that the warp stays converged; neighbours in LPT order are alike.
    auto fetch = [&](int last) -> int {
        if (W > 1 || !a.queue) return last < 0 ? (int)blockIdx.x * EPW : last + (int)gridDim.x * EPW;
        int v = 0;
        if (lane == 0) v = atomicAdd(a.queue, EPW);
        return __shfl_sync(kAll, v, 0);
    };
    for (int base = fetch(-1); base < a.N; base = fetch(base)) {
        const bool live = base + sub < a.N;
        const int slot = live ? base + sub : base;
        const int env = a.order ? __ldg(a.order + slot) : slot;
        int st = a.status[env];
        const float4 P0 = a.pose[2 * env], P1 = a.pose[2 * env + 1];
        const float4 V0 = a.vel[2 * env], V1 = a.vel[2 * env + 1];
        const float2 th = a.params[env];
        const int shp = a.shape[env];
        const int iters = a.iters[env];
        const int iters_w = wmax(iters);
        V3 x = xyz(P0);
        Q4 q = {P1.x, P1.y, P1.z, P1.w};
        V3 v = xyz(V0), w = xyz(V1);
        const float m = th.x, mu = th.y, inv_m = 1.0f / m;
        const int sfirst = __ldg(sc.shape_first + shp), NS = __ldg(sc.shape_count + shp);
        const int ncl = (NS + kCluster - 1) / kCluster;
        const float inv_ncl = 1.0f / (float)ncl;
        const int cfirst = __ldg(sc.cl_first + shp);
        int n_prev = 0;
        if (WARM) {   // the environment's impulse cache from its previous launch
            n_prev = a.cache_n[env];
#pragma unroll 1
            for (int k = gt; k < n_prev; k += E) prev[k] = a.cache[(size_t)env * cap + k];
        }
        double c_sum_env = (scored && gt == 0) ? a.c_sum[env] : 0.0;
        // cost of the frame just stepped against observation ob (Sec. III-C),
        // FP64 without contraction, pads in order; valid in the environment's first lane
        auto frame_cost = [&](const float *ob, int stt) -> double {
            const float inv_ns_f = 1.0f / (float)ns;
            sync();
            const double tau = (double)cfg.tau, wf = (double)cfg.w_force;
            const double tau2 = __dmul_rn(tau, tau);
#pragma unroll 1
            for (int p = gt; p < P; p += E) {
                const double fx = S.padacc[3 * p] * inv_ns_f, fy = S.padacc[3 * p + 1] * inv_ns_f,
                             fz = S.padacc[3 * p + 2] * inv_ns_f;
                const double ox = ob[3 * p], oy = ob[3 * p + 1], oz = ob[3 * p + 2];
                const double dx = __dsub_rn(fx, ox), dy = __dsub_rn(fy, oy), dz = __dsub_rn(fz, oz);
                const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                S.term[p] = __dmul_rn(wf, d2);
                const double ns2 = __dadd_rn(__dadd_rn(__dmul_rn(fx, fx), __dmul_rn(fy, fy)), __dmul_rn(fz, fz));
                const double no2 = __dadd_rn(__dadd_rn(__dmul_rn(ox, ox), __dmul_rn(oy, oy)), __dmul_rn(oz, oz));
                S.flag[p] = (ns2 > tau2) != (no2 > tau2);
            }
            sync();
            double c = 0.0;
            if (gt == 0) {
                if (stt & kDiverged) {
                    c = INFINITY;
                } else {
#pragma unroll 1
                    for (int p = 0; p < P; ++p) {
                        c = __dadd_rn(c, S.term[p]);
                        if (S.flag[p]) c = __dadd_rn(c, (double)cfg.w_contact);
                    }
                }
            }
            sync();   // S.term / S.flag are reused by the next frame
            return c;
        };

#pragma unroll 1
        for (int fr = 0; fr < a.n_frames; ++fr) {
#pragma unroll 1
            for (int k = gt; k < 3 * P; k += E) S.padacc[k] = 0.0f;
            const float4 *tab = a.link_tab + (size_t)(frame0 + fr) * (ns + 1) * Lk * kLinkStride;
            const bool act = live && (st & kDiverged) == 0;   // decided once per frame
            const int ns_w = __any_sync(kAll, act) ? ns : 0;
#pragma unroll 1
            for (int s = 0; s < ns_w; ++s) {
                const float4 *L0 = tab + (size_t)s * Lk * kLinkStride;
                const float4 *L1 = L0 + Lk * kLinkStride;
                const V3 v_pred = v + grav;
                const V3 w_pred = w;
                const M3 R = qmat(q);
                S6 Jb;   // inverse unit inertia, re-read (L1) rather than held in registers
                Jb.xx = __ldg(sc.shape_jinv + 6 * shp + 0); Jb.yy = __ldg(sc.shape_jinv + 6 * shp + 1);
                Jb.zz = __ldg(sc.shape_jinv + 6 * shp + 2); Jb.xy = __ldg(sc.shape_jinv + 6 * shp + 3);
                Jb.xz = __ldg(sc.shape_jinv + 6 * shp + 4); Jb.yz = __ldg(sc.shape_jinv + 6 * shp + 5);
                const S6 Wi = world_inv_inertia(R, Jb, inv_m);

                // -- 1. spheres and cluster centres to world (relative to x), cached
                //       (padding of the last cluster: far away); the links' offsets
#pragma unroll 1
                for (int j = gt; j < ncl * kCluster; j += E) {
                    float4 o = make_float4(kFar, kFar, kFar, 0.0f);
                    if (j < NS) {
                        const float4 sp = __ldg(sc.spheres + sfirst + j);
                        const V3 cr = mmul(R, xyz(sp));
                        o = make_float4(cr.x, cr.y, cr.z, sp.w);
                    }
                    sph[(j >> 3) * kSphStride + (j & 7)] = o;
                }
#pragma unroll 1
                for (int k = gt; k < ncl; k += E) {
                    const float4 cl = __ldg(sc.clusters + cfirst + k);
                    const V3 cr = mmul(R, xyz(cl));
                    clc[k] = make_float4(cr.x, cr.y, cr.z, cl.w);
                }
#pragma unroll 1
                for (int l = gt; l < Lk; l += E) {
                    const V3 xa = x - xyz(__ldg(L0 + l * kLinkStride));
                    const float4 ld = __ldg(L0 + l * kLinkStride + 1);
                    S.xa[l] = make_float4(xa.x, xa.y, xa.z, 0.0f);
                    S.ax[l] = ld;
                    S.lbeg[l] = 0;
                    S.lend[l] = 0;
                }
                sync();

                // -- 2a. cull (link, cluster) pairs by the clusters' enclosing spheres
                int nclp = 0;
                const int ncpairs = act ? Lk * ncl : 0, ncp_w = wmax(ncpairs);
#pragma unroll 2
                for (int p0 = 0; p0 < ncp_w; p0 += E) {
                    const int p = p0 + gt;
                    bool keep = false;
                    int e = 0;
                    if (p < ncpairs) {
                        const int l = min((int)(((float)p + 0.5f) * inv_ncl), Lk - 1), k = p - l * ncl;
                        const float4 cc = clc[k];
                        keep = cluster_reaches(sc, cfg, l, xyz(S.xa[l]) + xyz(cc), cc.w, xyz(S.ax[l]));
                        e = (l << 8) | k;
                    }
                    const int at = list(Int<1>{}, keep, nclp);
                    if (keep) clp[at] = (unsigned short)e;
                }
                sync();

                // -- 2b. a lane tests the eight spheres of a surviving pair
                int nc = 0;
                const int nclp_w = wmax(nclp);
#pragma unroll 1
                for (int e0 = 0; e0 < nclp_w; e0 += E) {
                    unsigned hits = 0;
                    int e = 0;
                    if (e0 + gt < nclp) {
                        e = clp[e0 + gt];
                        const int l = e >> 8, k = e & 0xff;
                        hits = cluster_hits(sc, cfg, l, k, xyz(S.xa[l]), xyz(S.ax[l]), sph + k * kSphStride, NS, inv_L);
                    }
                    const int idx = list(Int<4>{}, __popc(hits), nc);   // (0..8 a lane)
                    const int cj = (e & 0xff00) | ((e & 0xff) * kCluster);
#pragma unroll
                    for (int i = 0; i < kCluster; ++i) {
                        const int at = idx + __popc(hits & ((1u << i) - 1u));
                        if (((hits >> i) & 1u) && at < cap) clist[at] = (unsigned short)(cj + i);
                    }
                }
                sync();
                if (nc > cfg.c_max) {   // more contacts than the per-env capacity
                    st |= IH_ENV_OVERFLOW;
                    nc = 0;
                }
                if (act)   // the work counters, one lane each
                    work += gt == 0 ? nclp * kCluster : gt == 1 ? nc : gt == 2 ? nc * iters : gt == 3 ? 1 : gt == 4 ? (nc > 0 ? iters : 0) : ncpairs;

                // -- 3. contact setup, records to shared memory (past SC to the spill area);
                //       the contact range of each link
                const int nc_w = wmax(nc);
                const float trW = Wi.xx + Wi.yy + Wi.zz;
                auto setup = [&](int ci) {
                    const int e = clist[ci], l = e >> 8, j = e & 0xff;
                    const int e0 = ci > 0 ? clist[ci - 1] >> 8 : -1, e1 = ci < nc - 1 ? clist[ci + 1] >> 8 : -1;
                    if (e0 != l) S.lbeg[l] = (unsigned short)ci;
                    if (e1 != l) S.lend[l] = (unsigned short)(ci + 1);
                    const float4 sp = sph[(j >> 3) * kSphStride + (j & 7)];
                    const V3 cr = xyz(sp), ca = xyz(S.xa[l]) + cr;
                    const Hit hh = hit_link(sc, l, ca, sp.w, xyz(S.ax[l]), L0, inv_L);
                    const V3 r = cr - hh.n * sp.w;
                    cpad[ci] = PT.find(l, hh.t);
                    const CSetup cs = setup_contact(r, hh.n, hh.gap, l, Wi, trW, inv_m, cfg, L0, L1, x, inv_h);
                    const float4 r0 = make_float4(r.x, r.y, r.z, cs.ikt), r1 = make_float4(hh.n.x, hh.n.y, hh.n.z, cs.ikn),
                                 r2 = make_float4(cs.cc.x, cs.cc.y, cs.cc.z, 0.0f);
                    float4 l4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (WARM) {   // the pair's impulse at the end of the last substep (both lists are in pair order), else zero
                        int lo = 0, hi = n_prev;
#pragma unroll 1
                        while (lo < hi) {
                            const int mid = (lo + hi) >> 1;
                            if (__float_as_int(prev[mid].w) < e) lo = mid + 1; else hi = mid;
                        }
                        if (lo < n_prev && __float_as_int(prev[lo].w) == e) {
                            const float4 p4 = prev[lo];
                            l4 = make_float4(p4.x, p4.y, p4.z, 0.0f);
                        }
                    }
                    if (ci < RCAP) {
                        rec[3 * ci] = r0;
                        rec[3 * ci + 1] = r1;
                        rec[3 * ci + 2] = r2;
                        if (WARM) lamst[ci] = l4;
                    } else {
                        float4 *g4 = spill_g + (size_t)(ci - RCAP) * 4;
                        g4[0] = r0;
                        g4[1] = r1;
                        g4[2] = r2;
                        g4[3] = l4;
                    }
                };
#pragma unroll 1
                for (int ci = gt; ci < nc; ci += E) setup(ci);
                sync();   // (the impulses take the spheres' place)

                // -- 4. Jacobi projected-impulse iterations
                V3 vv = v_pred, ww = w_pred;
                if (nc_w > 0 && warp == 0) {
                    const float inv_nc = nc > 0 ? 1.0f / (float)nc : 0.0f, mu_s = 4096.0f * mu;
                    auto unpack = [&](Contact<float> &c, const float4 *c4, const float4 *l) {
                        const float4 s0 = c4[0], s1 = c4[1], s2 = c4[2];
                        c.r = {s0.x, s0.y, s0.z};
                        c.n = {s1.x, s1.y, s1.z};
                        c.c = {s2.x, s2.y, s2.z};
                        c.ikt = s0.w;
                        c.ikn = s1.w;
                        if (l) c.lam = {l->x, l->y, l->z};
                    };
                    // register slot k of the lane: contact gl + k L (empty past the list)
                    auto load1 = [&](Contact<float> &c, int k) {
                        const int ci = gl + k * L;
                        c.clear();
                        if (ci < nc) unpack(c, rec + 3 * ci, WARM ? lamst + ci : nullptr);
                    };
                    auto store1 = [&](float lx, float ly, float lz, int k) {
                        const int ci = gl + k * L;
                        if (ci < nc) lamst[ci] = make_float4(lx, ly, lz, 0.0f);
                    };
                    auto load2 = [&](Contact<F2> &c, int k) {
                        Contact<float> a, b;
                        load1(a, k);
                        load1(b, k + 1);
                        c.r = {{a.r.x, b.r.x}, {a.r.y, b.r.y}, {a.r.z, b.r.z}};
                        c.n = {{a.n.x, b.n.x}, {a.n.y, b.n.y}, {a.n.z, b.n.z}};
                        c.c = {{a.c.x, b.c.x}, {a.c.y, b.c.y}, {a.c.z, b.c.z}};
                        c.lam = {{a.lam.x, b.lam.x}, {a.lam.y, b.lam.y}, {a.lam.z, b.lam.z}};
                        c.ikn = {a.ikn, b.ikn};
                        c.ikt = {a.ikt, b.ikt};
                    };
                    auto store2 = [&](const Contact<F2> &c, int k) {
                        store1(c.lam.x.x, c.lam.y.x, c.lam.z.x, k);
                        store1(c.lam.x.y, c.lam.y.y, c.lam.z.y, k + 1);
                    };
                    // adds the wrenches of slots k (and k + 1) to their accumulators, slot mod NA, in slot order
                    auto add1 = [&](float (&acc)[NA][6], const Contact<float> &c, int k) {
                        float s[6];
                        c.wrench(s);
#pragma unroll
                        for (int q = 0; q < 6; ++q) acc[k % NA][q] += s[q];
                    };
                    auto add2 = [&](float (&acc)[NA][6], const Contact<F2> &c, int k) {
                        F2 s[6];
                        c.wrench(s);
#pragma unroll
                        for (int q = 0; q < 6; ++q) {
                            if constexpr (NA == 1) {
                                acc[0][q] = (acc[0][q] + s[q].x) + s[q].y;
                            } else {   // one packed addition
                                const F2 t = t_add(F2{acc[k % NA][q], acc[(k + 1) % NA][q]}, s[q]);
                                acc[k % NA][q] = t.x;
                                acc[(k + 1) % NA][q] = t.y;
                            }
                        }
                    };
                    auto body = [&](const float (&t)[6]) {
                        vv = v_pred + mk(t[0], t[1], t[2]) * inv_m;
                        const V3 mo = mk(t[3], t[4], t[5]);
                        if constexpr (WARM && TPE >= 64)   // (these instances' contraction: see prod_add)
                            ww = w_pred + mk(__fmaf_rn(Wi.xz, mo.z, prod_add(Wi.xy, mo.y, Wi.xx, mo.x)),
                                             __fmaf_rn(Wi.yz, mo.z, prod_add(Wi.yy, mo.y, Wi.xy, mo.x)),
                                             __fmaf_rn(Wi.zz, mo.z, prod_add(Wi.yz, mo.y, Wi.xz, mo.x)));
                        else
                            ww = w_pred + smul(Wi, mo);
                    };
                    if (WARM) {   // the cached impulses act from the first iteration on
                        float acc[NA][6] = {}, t[6];
#pragma unroll 1
                        for (int s0 = 0; s0 * L < nc_w; s0 += NA)
#pragma unroll
                            for (int j = 0; j < NA; ++j) {
                                const int ci = (s0 + j) * L + gl;
                                Contact<float> c;
                                c.clear();
                                if (ci < min(nc, RCAP)) unpack(c, rec + 3 * ci, lamst + ci);
                                else if (ci < nc) unpack(c, spill_g + (size_t)(ci - RCAP) * 4, spill_g + (size_t)(ci - RCAP) * 4 + 3);
                                add1(acc, c, j);
                            }
                        env_sum6<L, NA, NA>(acc, t, gl);
                        body(t);
                    }
                    // one loop per number of occupied slots, each a straight stretch of
                    // code: slots in pairs (packed), an odd last one alone. (Guarded slots in
                    // one loop kept the scheduler from interleaving them: 932 cycles an
                    // iteration at 1024 cylinders, 80 contacts.) Past its own count an
                    // environment of a 16-lane warp holds still (a step of zero)
                    auto rel = [&](int it) -> float { return (L == 32 || it < iters) ? inv_nc : 0.0f; };
                    auto iterate4 = [&](auto more) {
                        Contact<F2> c0, c2;
                        load2(c0, 0);
                        load2(c2, 2);
                        // FIRST: a lane's first further contact is read ahead and updated
                        // beside the register slots, in one stretch of code (an empty one
                        // adds zeros)
                        constexpr bool first = decltype(more)::value && FIRST;
                        float4 *g4 = nullptr;
                        if constexpr (first) {
                            g4 = spill_g + (size_t)gl * 4;
                            if (gl + RCAP >= nc) {
                                g4[0] = g4[2] = g4[3] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                                g4[1] = make_float4(0.0f, 0.0f, 1.0f, 0.0f);
                            }
                        }
#pragma unroll 1
                        for (int it = 0; it < iters_w; ++it) {
                            float acc[NA][6] = {}, t[6];
                            const float k = rel(it);
                            Contact<float> c4;
                            if constexpr (first) unpack(c4, g4, g4 + 3);
                            c0.update(vv, ww, mu_s, k);
                            c2.update(vv, ww, mu_s, k);
                            if constexpr (first) {
                                c4.update(vv, ww, mu_s, k);
                                g4[3] = make_float4(c4.lam.x, c4.lam.y, c4.lam.z, 0.0f);
                            }
                            add2(acc, c0, 0);
                            add2(acc, c2, 2);
                            if constexpr (first) add1(acc, c4, kSlots);
                            if constexpr (decltype(more)::value) {
#pragma unroll 1
                                for (int s0 = kSlots; (s0 + (first && s0 == kSlots)) * L < nc_w; s0 += NA)   // the (other) further ones, in the same per-thread order
#pragma unroll
                                    for (int j = 0; j < NA; ++j) {
                                        if (first && s0 + j == kSlots) continue;
                                        const int ci = (s0 + j) * L + gl;
                                        if (ci < nc) {
                                            float4 *g4 = spill_g + (size_t)(ci - RCAP) * 4;
                                            Contact<float> c;
                                            unpack(c, g4, g4 + 3);
                                            c.update(vv, ww, mu_s, k);
                                            g4[3] = make_float4(c.lam.x, c.lam.y, c.lam.z, 0.0f);
                                            add1(acc, c, j);
                                        }
                                    }
                            }
                            env_sum6<L, NA, NA>(acc, t, gl);
                            body(t);
                        }
                        store2(c0, 0);
                        store2(c2, 2);
                    };
                    if (nc_w <= L) {
                        Contact<float> c0;
                        load1(c0, 0);
#pragma unroll 1
                        for (int it = 0; it < iters_w; ++it) {
                            float acc[NA][6] = {}, t[6];
                            c0.update(vv, ww, mu_s, rel(it));
                            add1(acc, c0, 0);
                            env_sum6<L, NA, 1>(acc, t, gl);
                            body(t);
                        }
                        store1(c0.lam.x, c0.lam.y, c0.lam.z, 0);
                    } else if (nc_w <= 2 * L) {
                        Contact<F2> c0;
                        load2(c0, 0);
#pragma unroll 1
                        for (int it = 0; it < iters_w; ++it) {
                            float acc[NA][6] = {}, t[6];
                            c0.update(vv, ww, mu_s, rel(it));
                            add2(acc, c0, 0);
                            env_sum6<L, NA, (NA < 2 ? NA : 2)>(acc, t, gl);
                            body(t);
                        }
                        store2(c0, 0);
                    } else if (nc_w <= 3 * L) {
                        Contact<F2> c0;
                        Contact<float> c2;
                        load2(c0, 0);
                        load1(c2, 2);
#pragma unroll 1
                        for (int it = 0; it < iters_w; ++it) {
                            float acc[NA][6] = {}, t[6];
                            const float k = rel(it);
                            c0.update(vv, ww, mu_s, k);
                            c2.update(vv, ww, mu_s, k);
                            add2(acc, c0, 0);
                            add1(acc, c2, 2);
                            env_sum6<L, NA, (NA < 3 ? NA : 3)>(acc, t, gl);
                            body(t);
                        }
                        store2(c0, 0);
                        store1(c2.lam.x, c2.lam.y, c2.lam.z, 2);
                    } else if (nc_w <= kSlots * L) {
                        iterate4(Flag<false>{});
                    } else {
                        iterate4(Flag<true>{});
                    }
                }
                if constexpr (W > 1) {   // the body's velocity to the team's other warps
                    if (threadIdx.x == 0) {
                        S.fin[0] = vv.x; S.fin[1] = vv.y; S.fin[2] = vv.z;
                        S.fin[3] = ww.x; S.fin[4] = ww.y; S.fin[5] = ww.z;
                    }
                    sync();
                    vv = mk(S.fin[0], S.fin[1], S.fin[2]);
                    ww = mk(S.fin[3], S.fin[4], S.fin[5]);
                }

                // -- 5. symplectic Euler with the exact rotation exponential
                if (act) {
                    v = vv;
                    w = ww;
                    x = x + v * h;
                    const float wn = sqrtf(dot(w, w));
                    float sn, cs;
                    sincosf(0.5f * wn * h, &sn, &cs);
                    const float kq = (wn > 0.0f) ? sn / wn : 0.5f * h;
                    q = qnorm(qmul({cs, w.x * kq, w.y * kq, w.z * kq}, q));
                }
                // sensor pads: force on the pad by the object is -lambda / h, summed
                // over the contacts of the pad's link in contact order
                __syncwarp();
#pragma unroll 1
                for (int k = gt; k < 3 * P; k += E) {
                    const int p = k / 3, comp = k - 3 * p;
                    const int l = __ldg(sc.pad_link + p);
                    float f = 0.0f;
                    const int e = S.lend[l], es = min(e, RCAP);
                    int ci = S.lbeg[l];
                    const float *lc = reinterpret_cast<const float *>(lamst) + comp;
#pragma unroll 4
                    for (; ci < es; ++ci) f -= (cpad[ci] == p ? lc[4 * ci] : 0.0f) * inv_h;
#pragma unroll 1
                    for (; ci < e; ++ci) f -= (cpad[ci] == p ? reinterpret_cast<const float *>(spill_g + (size_t)(ci - RCAP) * 4 + 3)[comp] : 0.0f) * inv_h;
                    S.padacc[k] += f;
                }
                if (WARM) {   // this substep's contacts and final impulses, for the next one
#pragma unroll 1
                    for (int ci = gt; ci < nc; ci += E) {
                        const float4 l3 = ci < RCAP ? lamst[ci] : spill_g[(size_t)(ci - RCAP) * 4 + 3];
                        prev[ci] = make_float4(l3.x, l3.y, l3.z, __int_as_float(clist[ci]));
                    }
                    if (act) n_prev = nc;
                }
                sync();
            }
            if (act) {
                if (!all_finite(x, q, v, w)) st |= IH_ENV_NONFINITE;
                else if (dot(x, x) > cfg.escape_radius * cfg.escape_radius) st |= IH_ENV_ESCAPED;
            }
            if (scored) {   // this frame's cost, window sum and mean (every frame, or a single one); the frame's pose
                const double c = frame_cost(obs + (size_t)fr * P * 3, st);
                if (gt == 0 && live) {
                    c_sum_env = __dadd_rn(c_sum_env, c);
                    double cm = __ddiv_rn(c_sum_env, (double)(n_win0 + fr + 1));
                    if (window_mode) {
                        a.cm_frames[(size_t)fr * a.N + env] = cm;
                        float4 *pf = a.pose_frames + 2 * ((size_t)fr * a.N + env);
                        pf[0] = make_float4(x.x, x.y, x.z, 0.0f);
                        pf[1] = make_float4(q.w, q.x, q.y, q.z);
                    }
                    if (fr == a.n_frames - 1) {
                        a.c_sum[env] = c_sum_env;
                        a.c_mean[env] = cm;
                        if (a.cost_mean) a.cost_mean[env] = cm;
                        const unsigned long long key = cost_key(isnan(cm) ? INFINITY : cm);
                        if (key < best_k || (key == best_k && env < best_i)) { best_k = key; best_i = env; }
                    }
                }
            }
        }
        // forces of the last frame, averaged over its substeps
        const float inv_ns = 1.0f / (float)ns;
        float *fo = a.forces + (size_t)env * P * 3;
        sync();
#pragma unroll 1
        for (int k = gt; k < 3 * P && live; k += E) fo[k] = S.padacc[k] * inv_ns;
        if (gt == 0 && live) {
            a.pose[2 * env] = make_float4(x.x, x.y, x.z, 0.0f);
            a.pose[2 * env + 1] = make_float4(q.w, q.x, q.y, q.z);
            a.vel[2 * env] = make_float4(v.x, v.y, v.z, 0.0f);
            a.vel[2 * env + 1] = make_float4(w.x, w.y, w.z, 0.0f);
            a.status[env] = st;
        }
        if (WARM && live) {   // the cache for the next launch
            if (gt == 0) a.cache_n[env] = n_prev;
#pragma unroll 1
            for (int k = gt; k < n_prev; k += E) a.cache[(size_t)env * cap + k] = prev[k];
        }
        sync();
    }
    if (gt < 6 && a.work && work) atomicAdd(a.work + gt, work);
    if (a.queue && threadIdx.x == 0) {   // the last block to finish empties the queue for the next launch
        __threadfence();   // this block's queue draws, before its finish ticket
        if (atomicAdd(a.queue + 1, 1) == (int)gridDim.x - 1) {
            atomicExch(a.queue, 0);
            atomicExch(a.queue + 1, 0);
        }
    }
    if (!scored || window_mode || warp > 0) return;
    // argmin (C_i, i) over the grid: per-block candidate, then the last block
    auto better = [&](unsigned long long k, int i) {
        if (k < best_k || (k == best_k && i < best_i)) { best_k = k; best_i = i; }
    };
    if (L == 16) better(__shfl_sync(kAll, best_k, 16), __shfl_sync(kAll, best_i, 16));
    bool last = false;
    __threadfence();   // this thread's pose/status/cost writes, before the ticket
    __syncwarp();
    if (lane == 0) {
        a.part_c[blockIdx.x] = __longlong_as_double((long long)best_k);
        a.part_i[blockIdx.x] = best_i;
        __threadfence();
        last = atomicAdd(a.done, 1u) == gridDim.x - 1;
    }
    if (!__shfl_sync(kAll, (int)last, 0)) return;
    __threadfence();
    best_k = ~0ull;
    best_i = 0x7fffffff;
#pragma unroll 4
    for (int b = lane; b < (int)gridDim.x; b += 32)
        better((unsigned long long)__double_as_longlong(__ldcg(a.part_c + b)), __ldcg(a.part_i + b));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) better(__shfl_xor_sync(kAll, best_k, o), __shfl_xor_sync(kAll, best_i, o));
    const int best = (best_i == 0x7fffffff) ? 0 : best_i;
    if (lane == 0) {
        int *argmin_out = a.argmin_out;
        if (a.win) argmin_out = a.win->argmin ? a.win->argmin + a.win_k : nullptr;
        *a.argmin_state = best;
        if (argmin_out) *argmin_out = best;
        *a.n_window = n_win0 + 1;
        *a.done = 0u;
    }
    float *est_out = a.est_pose_out;
    if (a.win) est_out = a.win->est ? a.win->est + 8 * a.win_k : nullptr;
    if (est_out && lane < 8) {
        const float4 p = __ldcg(a.pose + 2 * best + (lane >> 2));
        const float v[4] = {p.x, p.y, p.z, p.w};
        est_out[lane] = v[lane & 3];
    }
}

template <int L, int TPE, bool WARM>
size_t bytes_t(int s_max, int c_max, int clp_cap) {
    return sizeof(PadTable) + 32 / L * env_bytes(s_max, stage_capacity(L, c_max), c_max, WARM, clp_cap);
}

// Shared-memory opt-in, and the blocks of this kernel that fit on one SM
template <int L, int TPE, bool WARM, int B, bool FIRST, int W>
cudaError_t prepare_t(int s_max, int c_max, int clp_cap, int *blocks_per_sm) {
    const size_t bytes = bytes_t<L, TPE, WARM>(s_max, c_max, clp_cap);
    cudaError_t e = cudaSuccess;
    if (bytes > 48 * 1024)
        e = cudaFuncSetAttribute(step_kernel<L, TPE, WARM, B, FIRST, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && blocks_per_sm)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, step_kernel<L, TPE, WARM, B, FIRST, W>, 32 * W, bytes);
    return e;
}

// The dispatch over the compiled kernels, for the cold (WARM = false) or the
// warm-started (WARM = true) solver; each is instantiated in its own
// translation unit so the two build in parallel.
template <bool WARM>
cudaError_t prepare_w(const StepVariant &v, int s_max, int c_max, int clp_cap, int *blocks_per_sm) {
#define IH_PREP(L, T, B, F, W)                                                              \
    if (v.lanes == L && v.group == T && v.per_sm == B && v.first == F && v.warps == W)      \
        return prepare_t<L, T, WARM, B, F, W>(s_max, c_max, clp_cap, blocks_per_sm);
    IH_STEP_KERNELS(IH_PREP)
#undef IH_PREP
    return cudaErrorInvalidValue;
}

template <bool WARM>
cudaError_t launch_w(const StepArgs &a, const StepVariant &v, int grid, int s_max, cudaStream_t s) {
#define IH_LAUNCH(L, T, B, F, W)                                                                                                \
    if (v.lanes == L && v.group == T && v.per_sm == B && v.first == F && v.warps == W) {                                        \
        step_kernel<L, T, WARM, B, F, W><<<grid, 32 * W, bytes_t<L, T, WARM>(s_max, a.cfg.c_max, a.clp_cap), s>>>(a, s_max);    \
        return cudaGetLastError();                                                                                              \
    }
    IH_STEP_KERNELS(IH_LAUNCH)
#undef IH_LAUNCH
    return cudaErrorInvalidValue;
}

}  // namespace
}  // namespace ih
