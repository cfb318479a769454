"""Measured cases: the calls a tracking program makes, over the sizes it makes them at.

A case names a workload of `paper_2002_12160_gb300.workloads` (the parity, tracking,
uneven-batch and throughput configurations of this repository), a number of
environments and a number of frames, and what the program does with them:

  frames  a resumed population is stepped and scored for T frames (Algorithm 1's inner
          loop): `sim_step_track` for a single frame, else `sim_step_frames` and
          `sim_frames_argmin`
  window  a whole tracking window: `sim_track_window` (frames, argmin, elite resample)
  calls   the same loop as separate calls, one frame and one update: `sim_step`,
          `sim_read_sensors`, `cost_eval`, `optimizer_update`
  grad    gradient of the horizon cost: `autograd.tracking_cost` and its backward for a
          whole batch, `sim_adjoint` for chosen environments (the elites a refinement takes)
  pd      T frames of the PD-driven hand scored with the full cost: `sim_step_frames_full`
          and `sim_frames_argmin`

Every pass starts from the same population, handed over with `sim_set_state`. The
populations are grasps in progress: a few hundred environments simulated here, in FP64
torch, from the initial sampling until the fingers have closed, then copied with the
optimizer's exploration noise, which is what a window starts from after a resample.
`exact` is the same FP64 torch simulation of the case itself.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2002_12160_gb300 import autograd, inhand, workloads as W

WARM_FROM, F0 = 8, 16      # simulated lead-in: frames [8, 16), the case starts at frame 16
BASE = 256                 # environments of the lead-in
F64 = torch.float64


def listed():
    return [
        # the smallest call: the 16-environment parity configuration, one control tick
        dict(name="box 16 frame", kind="frames", workload="tracking_box27", n=16, frames=1),
        # the tracking configuration's window, without the optimizer
        dict(name="cylinder 1024 frames", kind="frames", workload="tracking_cyl64", n=1024, frames=10),
        # the warm-started solver at few iterations, a box population
        dict(name="box 1000 warm frames", kind="frames", workload="tracking_box27", n=1000, frames=10, warm=True, iters=10),
        # uneven shapes and iteration counts in one batch
        dict(name="uneven 8192 frames", kind="frames", workload="uneven_mixed", n=8192, frames=10),
        # the throughput sweep's largest batch: 4 substeps, 40 iterations
        dict(name="mug 32768 frames", kind="frames", workload="sweep_mug128", n=32768, frames=2),
        # the whole tracking call
        dict(name="cylinder 1024 window", kind="window", workload="tracking_cyl64", n=1024, frames=10),
        # the paper's loop call by call, REPS draws with replacement
        dict(name="box 4096 calls", kind="calls", workload="tracking_box27", n=4096, frames=1, opt="reps"),
        # a small differentiable batch through autograd
        dict(name="box 64 gradient", kind="grad", workload="tracking_box27", n=64, frames=5),
        # the elites of a 1024-environment tracker over its window (what a refinement step evaluates)
        dict(name="cylinder 102 gradient", kind="grad", workload="tracking_cyl64", n=1024, frames=10, envs=102),
        # the differentiable-tracking configuration: a 30-frame horizon, checkpoints every 10
        dict(name="cylinder 1024 gradient", kind="grad", workload="tracking_cyl64", n=1024, frames=30),
        # the PD-driven hand's window with the full observation and cost
        dict(name="cylinder 1024 pd", kind="pd", workload="tracking_cyl64", n=1024, frames=10),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["frames", "frames", "frames", "window", "calls", "grad", "pd"])
    if kind == "frames":
        name = rng.choice(["tracking_box27", "tracking_cyl64", "uneven_mixed", "sweep_mug128"])
        n = size(16, 32768 if name == "sweep_mug128" else 8192)
        frames = rng.randint(1, 2 if n > 8192 else 10 if name != "sweep_mug128" else min(10, max(1, 65536 // n)))
        c = dict(kind=kind, workload=name, n=n, frames=frames)
        if name in ("tracking_box27", "tracking_cyl64") and rng.random() < 0.4:
            c.update(warm=True, iters=rng.choice([5, 10, 20]))
        return c
    if kind == "window":
        return dict(kind=kind, workload=rng.choice(["tracking_box27", "tracking_cyl64"]), n=size(64, 8192),
                    frames=rng.randint(5, 10), opt=rng.choice(["elite", "wrs", "reps"]))
    if kind == "calls":
        return dict(kind=kind, workload=rng.choice(["tracking_box27", "tracking_cyl64"]), n=size(64, 16384), frames=1,
                    opt=rng.choice(["elite", "wrs", "reps"]))
    if kind == "grad":
        name = rng.choice(["tracking_box27", "tracking_cyl64"])
        n = size(8, 1024)
        c = dict(kind=kind, workload=name, n=n, frames=rng.randint(3, 30))
        if rng.random() < 0.4:
            c["envs"] = max(1, n // 10)
        return c
    return dict(kind=kind, workload=rng.choice(["tracking_box27", "tracking_cyl64"]), n=size(32, 2048),
                frames=rng.randint(1, 10))


# ---------------------------------------------------------------- FP64 torch simulation
def qmul(a, b):
    aw, ax, ay, az = a.unbind(-1)
    bw, bx, by, bz = b.unbind(-1)
    return torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                        aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], -1)


def qexp(w):
    t2 = (w * w).sum(-1, keepdim=True)
    t = torch.sqrt(t2 + 1e-60)
    return torch.cat([torch.cos(0.5 * t), w * torch.where(t2 > 1e-24, torch.sin(0.5 * t) / t, 0.5 + 0 * t)], -1)


def qmat(q):
    w, x, y, z = q.unbind(-1)
    return torch.stack([torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)], -1),
                        torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)], -1),
                        torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1)], -2)


def dot(a, b):
    return (a * b).sum(-1, keepdim=True)


def cross(a, b):
    return torch.linalg.cross(*torch.broadcast_tensors(a, b))


def mv(M, v):   # matrices [..., 3, 3] on vectors [..., 3]
    return (M * v[..., None, :]).sum(-1)


class SoftNormal(torch.autograd.Function):
    """max(0, z), with the derivative sigmoid(beta z)."""

    @staticmethod
    def forward(ctx, z, beta):
        ctx.save_for_backward(z)
        ctx.beta = beta
        return z.clamp(min=0)

    @staticmethod
    def backward(ctx, g):
        return g * torch.sigmoid(ctx.beta * ctx.saved_tensors[0]), None


class SoftDisk(torch.autograd.Function):
    """z clamped radially to |z| <= L, with the derivative of z smin(|z|, L) / |z|."""

    @staticmethod
    def forward(ctx, z, L, width):
        ctx.save_for_backward(z, L)
        ctx.width = width
        t2 = dot(z, z)
        return torch.where(t2 > L * L, z * (L / torch.sqrt(t2 + 1e-300)), z)

    @staticmethod
    def backward(ctx, g):
        z, L = ctx.saved_tensors
        w = ctx.width
        a = torch.sqrt(dot(z, z))
        zero = a == 0
        a = torch.where(zero, torch.ones_like(a), a)
        Q = torch.sqrt((a - L) ** 2 + (w * L) ** 2)
        phi = L * (4 * a - w * w * L) / (2 * (a + L + Q))
        pa, pb = 0.5 * (1 - (a - L) / Q), 0.5 * (1 + ((a - L) - w * w * L) / Q)
        zh = z / a
        s = dot(zh, g)
        gz = torch.where(zero, torch.where(L > 0, g, torch.zeros_like(g)), g * (phi / a) + zh * (s * (pa - phi / a)))
        return gz, torch.where(zero, torch.zeros_like(s), s * pb), None


class Reference:
    """The frame step of a workload for a batch, in FP64."""

    def __init__(self, wl, shape, iters, dev, smooth=None):
        f = lambda a: torch.as_tensor(np.asarray(np.asarray(a, np.float32), np.float64), dtype=F64, device=dev)
        sc, self.cfg, self.dev, self.smooth = wl.scene, wl.sim, dev, smooth
        self.sc = sc
        S = max(len(s) for s in sc.shapes)
        body, rad = torch.zeros(len(sc.shapes), S, 3, dtype=F64, device=dev), -torch.ones(len(sc.shapes), S, dtype=F64, device=dev)
        Ji = []
        for k, rows in enumerate(sc.shapes):
            r = np.asarray(np.asarray(rows, np.float32), np.float64)
            c = r[:, :3] - r[:, :3].mean(0)
            body[k, :len(r)], rad[k, :len(r)] = (torch.as_tensor(a, device=dev) for a in (c, r[:, 3]))
            # equal solid balls about the centroid
            J = np.mean(0.4 * r[:, 3] ** 2 + (c * c).sum(1)) * np.eye(3) - c.T @ c / len(r)
            Ji.append(torch.as_tensor(np.linalg.inv(J), device=dev))
        shape = torch.as_tensor(np.asarray(shape), dtype=torch.long, device=dev)
        self.body, self.rad, self.Ji, self.S = body[shape], rad[shape], torch.stack(Ji)[shape], S
        self.iters = torch.as_tensor(np.asarray(iters), device=dev)
        self.half, self.root, self.Lk = f(sc.palm_half), f(sc.finger_root), sc.n_links
        self.len, self.lrad = float(np.float32(sc.link_len)), float(np.float32(sc.link_rad))
        c32 = lambda v: float(np.float32(v))
        self.h = c32(self.cfg.frame_dt) / self.cfg.substeps
        self.margin, self.beta, self.slop = c32(self.cfg.margin), c32(self.cfg.beta), c32(self.cfg.slop)
        self.g = f(self.cfg.gravity)
        self.q = torch.as_tensor(wl.q_traj, device=dev).to(F64)
        s0, s1 = f(sc.pad_s0), f(sc.pad_s1)
        self.pad_link = torch.as_tensor(np.asarray(sc.pad_link), device=dev)
        self.s0, self.s1 = torch.where(self.pad_link == 0, -1, s0), torch.where((self.pad_link == 0) | (s1 >= 1), 2, s1)
        if self.cfg.hand != "pd":   # the commanded hand at every substep boundary
            ns = self.cfg.substeps
            frac = torch.arange(ns + 1, dtype=F64, device=dev)[:, None] / ns
            at = self.q[:-1, None] + frac * (self.q[1:, None] - self.q[:-1, None])
            lp, lq, _, _ = self.fk(at.reshape(-1, at.shape[-1]))
            self.tab = [v.reshape(-1, ns + 1, *v.shape[1:]) for v in (lp, lq, qmat(lq))]
        else:
            self.kp, self.kd, self.arm = c32(self.cfg.kp), c32(self.cfg.kd), c32(self.cfg.armature)
            self.M = self.arm + self.h * self.kd + self.h ** 2 * self.kp

    def fk(self, q):
        """Joint angles [B, D] -> link positions [B, Lk, 3], quaternions [B, Lk, 4], joint axes and origins [B, D, 3]."""
        B, F = q.shape[0], self.sc.n_fingers
        q = q.reshape(B, F, 4)
        zero, one = torch.zeros(B, F, 1, dtype=F64, device=self.dev), torch.ones(B, F, 1, dtype=F64, device=self.dev)
        turn = lambda ang, z: torch.cat([torch.cos(ang / 2), *((zero, zero, torch.sin(ang / 2)) if z else (zero, torch.sin(ang / 2), zero))], -1)
        p = self.root[:, :3].expand(B, F, 3)
        r = qmul(turn(self.root[:, 3:] + q[..., :1], True), turn(-0.5 * math.pi * one, False))
        pos, quat, zax, org = [p], [r], [torch.cat([zero, zero, one], -1)], [p]
        for j in range(1, 4):
            R = qmat(r)
            p = p + R[..., 0] * self.len
            r = qmul(r, turn(-q[..., j:j + 1], False))
            pos.append(p), quat.append(r), zax.append(-R[..., 1]), org.append(p)
        palm = torch.cat([one[:, :1], zero[:, :1], zero[:, :1], zero[:, :1]], -1)
        flat = lambda v: torch.stack(v, 2).reshape(B, 4 * F, -1)
        return torch.cat([0 * palm[..., :3], flat(pos)], 1), torch.cat([palm, flat(quat)], 1), flat(zax), flat(org)

    def narrow(self, c, rad, a, R, palm):
        """Gap, normal and axial fraction of spheres against their links (a, R; palm: the box, else a capsule)."""
        ca = c - a
        u = R[..., 0]
        tr = dot(ca, u) / self.len
        t = tr.clamp(0, 1)
        diff = ca - u * (t * self.len)
        dist = torch.sqrt(dot(diff, diff) + 1e-300)
        cl = mv(R.transpose(-1, -2), ca)
        k = torch.maximum(torch.minimum(cl, self.half), -self.half)
        inside = (k == cl).all(-1, keepdim=True)
        db = cl - k
        distb = torch.sqrt(dot(db, db) + 1e-300)
        face = torch.stack([self.half[0] - cl[..., 0], self.half[0] + cl[..., 0], self.half[1] - cl[..., 1],
                            self.half[1] + cl[..., 1], self.half[2] - cl[..., 2], self.half[2] + cl[..., 2]], -1)
        best = face.detach().argmin(-1, keepdim=True)
        nl = torch.zeros_like(cl).scatter(-1, best // 2, (1 - 2 * (best % 2)).to(F64))
        gapb = torch.where(inside, -face.gather(-1, best), distb)
        nb = mv(R, torch.where(inside, nl, db / distb))
        gap = torch.where(palm, gapb, dist - self.lrad) - rad
        return gap, torch.where(palm, nb, diff / dist), torch.where(palm, torch.zeros_like(t), t)

    def pairs(self, x, cr, a, R):
        """Indices [N, C] of the pairs within the margin (link * S + sphere) and which entries are used."""
        N = x.shape[0]
        c = (x[:, None] + cr)[:, None]
        hits, many = [], max(1, int(2e7) // (N * self.S))
        for l in range(0, self.Lk, many):   # a few links at a time, to bound the memory
            palm = torch.arange(l, min(l + many, self.Lk), device=self.dev)[:, None, None] == 0
            gap, _, _ = self.narrow(c, self.rad[:, None, :, None], a[:, l:l + many, None], R[:, l:l + many, None], palm)
            hits.append((gap[..., 0] < self.margin) & (self.rad > 0)[:, None])
        hit = torch.cat(hits, 1).reshape(N, -1)
        nc = hit.sum(1)
        hit &= (nc <= self.cfg.c_max)[:, None]
        C = max(1, int(hit.sum(1).max()))
        e, p = hit.nonzero(as_tuple=True)
        k = hit.cumsum(1)[e, p] - 1
        idx = torch.zeros(N, C, dtype=torch.long, device=self.dev)
        on = torch.zeros(N, C, dtype=torch.bool, device=self.dev)
        idx[e, k], on[e, k] = p, True
        return idx, on, nc > self.cfg.c_max

    def substep(self, st, m, mu, f, s, forces):
        x, q, v, w = st["x"], st["q"], st["v"], st["w"]
        h, ns, pd = self.h, self.cfg.substeps, self.cfg.hand == "pd"
        N = x.shape[0]
        u0, u1 = self.q[f], self.q[f + 1]
        if pd:
            lp, lq, zax, org = self.fk(st["qj"])
            lR = qmat(lq)
            qds = (self.arm * st["qd"] + h * self.kp * (u0 + (s + 1) / ns * (u1 - u0) - st["qj"])) / self.M
        else:
            lp, lR, lp1, lR1 = (self.tab[k][f, s + d, None] for d in (0, 1) for k in (0, 2))
        vp = v + h * self.g
        R = qmat(q)
        Wi = R @ self.Ji @ R.transpose(-1, -2) / m[..., None]
        cr = mv(R[:, None], self.body)
        with torch.no_grad():
            idx, on, over = self.pairs(x, cr, lp, lR)
        sp, l = idx % self.S, idx // self.S
        e = torch.arange(N, device=self.dev)[:, None]
        b = e if pd else torch.zeros_like(e)
        crc = mv(R[:, None], self.body[e, sp])
        rad = self.rad[e, sp][..., None]
        A, RA = lp[b, l], lR[b, l]
        gap, n, t = self.narrow(x[:, None] + crc, rad, A, RA, (l == 0)[..., None])
        r = crc - n * rad
        of = on[..., None].to(F64)
        rn, W4 = cross(r, n), Wi[:, None]
        kn = 1 / m[:, None] + dot(rn, mv(W4, rn))
        trK = 3 / m[:, None] + dot(r, r) * Wi.diagonal(dim1=-2, dim2=-1).sum(-1)[:, None, None] - dot(r, mv(W4, r))
        bias = torch.where(gap > 0, gap / h, (self.beta * (gap + self.slop).clamp(max=0) / h).clamp(min=-self.cfg.vmax))
        if pd:
            ja = torch.arange(self.sc.n_joints, device=self.dev)
            moves = (l[..., None] >= 1) & (ja // 4 == (l[..., None] - 1) // 4) & (ja % 4 <= (l[..., None] - 1) % 4)
            J = cross(zax[:, None], (x[:, None] + r)[:, :, None] - org[:, None]) * (moves & on[..., None])[..., None]
            kn = kn + (dot(J, n[:, :, None])[..., 0] ** 2).sum(-1, keepdim=True) / self.M
            trK = trK + (J * J).sum((-1, -2))[..., None] / self.M
            vl = (J * qds[:, None, :, None]).sum(2)
        else:
            p = x[:, None] + r
            pl = mv(RA.transpose(-1, -2), p - A)
            vl = ((lp1[b, l] - A) + (mv(lR1[b, l], pl) - mv(RA, pl))) / h * (l > 0)[..., None]
        ikn, ikt = of / kn, of * 2 / (trK - kn)
        nc = on.sum(1).clamp(min=1).to(F64)[:, None, None]
        lam = torch.zeros_like(r)
        vv, ww, qd = vp, w, qds if pd else None
        for it in range(int(self.iters.max())):
            u = vv[:, None] + cross(ww[:, None], r) - (vl - n * bias)
            un, lo = dot(u, n), dot(lam, n)
            zn, zt = lo - un * ikn, (lam - n * lo) - (u - n * un) * ikt
            if self.smooth:
                ln = SoftNormal.apply(zn, self.smooth[0])
                lt = SoftDisk.apply(zt, mu[:, None] * ln, self.smooth[1])
            else:
                ln = zn.clamp(min=0)
                t2, lim = dot(zt, zt), mu[:, None] * ln
                lt = torch.where(t2 > lim * lim, zt * (lim / torch.sqrt(t2 + 1e-300)), zt)
            go = (it < self.iters)[:, None, None]
            lam = torch.where(go, lam + (n * ln + lt - lam) / nc * of, lam)
            vv = vp + lam.sum(1) / m
            ww = w + mv(Wi, cross(r, lam).sum(1))
            if pd:
                qd = qds - (J * lam[:, :, None]).sum((1, 3)) / self.M
                vl = (J * qd[:, None, :, None]).sum(2)
        # the first pad of the contact's link whose interval holds t
        t0 = t.detach()
        holds = (self.pad_link == l[..., None]) & on[..., None] & (t0 >= self.s0) & (t0 < self.s1)
        which = (holds & (holds.cumsum(-1) == 1)).to(F64)
        forces = forces - (which[..., None] * lam[:, :, None]).sum(1) / h
        qn = qmul(qexp(ww * h), q)
        new = dict(x=x + vv * h, q=qn / torch.sqrt(dot(qn, qn)), v=vv, w=ww)
        if pd:
            new.update(qd=qd, qj=st["qj"] + h * qd)
        return new, forces, over

    def frame(self, st, m, mu, f, dead):
        """One frame; `dead` environments keep their state and report no force."""
        forces = torch.zeros(st["x"].shape[0], self.sc.n_pads, 3, dtype=F64, device=self.dev)
        new, over = st, dead.clone()
        for s in range(self.cfg.substeps):
            new, forces, o = self.substep(new, m, mu, f, s, forces)
            over = over | o
        keep = dead[:, None]
        new = {k: torch.where(keep, st[k], a) for k, a in new.items()}
        forces = torch.where(keep[..., None], torch.zeros_like(forces), forces / self.cfg.substeps)
        return new, forces, over | (dot(new["x"], new["x"])[:, 0] > self.cfg.escape_radius ** 2)


def state_of(ten, pd):
    d = {k: v.to(F64) for k, v in ten.items() if torch.is_tensor(v) and v.is_floating_point()}
    st = dict(x=d["pose"][:, :3], q=d["pose"][:, 4:8], v=d["vel"][:, :3], w=d["vel"][:, 4:7])
    if pd:
        st.update(qj=d["qj"], qd=d["qd"])
    return st, d["params"][:, :1], d["params"][:, 1:]


def pose8(x, q):
    return torch.cat([x, torch.zeros_like(x[:, :1]), q], 1)


def vel8(v, w):
    z = torch.zeros_like(v[:, :1])
    return torch.cat([v, z, w, z], 1)


# ---------------------------------------------------------------- inputs
def make_workload(case, seed):
    frames = F0 + case["frames"] + 1
    wl = W.make_workload(case["workload"], n_envs=case["n"], frames=frames, seed=100003 + seed)
    sim = dataclasses.replace(wl.sim, warm_start=bool(case.get("warm", False)), iters=case.get("iters", wl.sim.iters),
                              hand="pd" if case["kind"] == "pd" else "kinematic")
    wl.sim = sim
    if "iters" in case:
        wl.iters[:] = case["iters"]
    wl.opt = dataclasses.replace(wl.opt, kind=case.get("opt", "elite"))
    return wl


def inputs(case, seed):
    """(workload, tensors): the population at the start of frame F0 and the true environment's observations."""
    wl = make_workload(case, seed)
    dev = torch.device("cuda")
    rng = np.random.default_rng(seed * 7919 + 13)
    n, pd = case["n"], case["kind"] == "pd"
    B = min(n, BASE)
    sid = wl.shape_id[:B]
    # the lead-in: the initial sampling, stepped with few iterations until the fingers have closed;
    # its last environment is the true one
    nom = np.stack([W.nominal_pose_for(wl.scene, k) for k in range(len(wl.scene.shapes))])
    pose = nom[np.append(sid, 0)].astype(np.float64)
    rot = rng.normal(0, wl.init.sigma_r, (B + 1, 3))
    pose[:, :3] += rng.normal(0, wl.init.sigma_p, (B + 1, 3))
    par = np.column_stack([rng.uniform(*wl.init.m_range, B + 1), rng.uniform(*wl.init.mu_range, B + 1)])
    t = lambda a: torch.as_tensor(a, dtype=F64, device=dev)
    lead = dataclasses.replace(wl, sim=dataclasses.replace(wl.sim, iters=8, substeps=2))
    ref = Reference(lead, np.append(sid, 0), np.full(B + 1, 8), dev)
    st = dict(x=t(pose[:, :3]), q=qexp(t(rot)), v=torch.zeros(B + 1, 3, dtype=F64, device=dev),
              w=torch.zeros(B + 1, 3, dtype=F64, device=dev))
    if pd:
        st.update(qj=ref.q[WARM_FROM].expand(B + 1, -1).clone(), qd=torch.zeros(B + 1, wl.scene.n_joints, dtype=F64, device=dev))
    m, mu = t(par[:, :1]), t(par[:, 1:])
    dead = torch.zeros(B + 1, dtype=torch.bool, device=dev)
    for f in range(WARM_FROM, F0):
        st, _, dead = ref.frame(st, m, mu, f, dead)
    # the population: copies of the lead-in's environments of the same shape, explored by the
    # optimizer's floor; the first tenth unexplored, as elites
    of_shape = {k: np.flatnonzero(sid == k) for k in np.unique(wl.shape_id)}
    parent = np.array([rng.choice(of_shape[k]) if len(of_shape[k]) else 0 for k in wl.shape_id], np.int64)
    floor = np.asarray(wl.opt.floor_std) * (np.arange(n)[:, None] >= n // 10)
    dz = t(rng.normal(0, 1, (n, 8)) * floor)
    pt = torch.as_tensor(parent, device=dev)
    ten = dict(pose=pose8(st["x"][pt] + dz[:, :3], qmul(qexp(dz[:, 3:6]), st["q"][pt])).float(), vel=vel8(st["v"][pt], st["w"][pt]).float(),
               params=torch.cat([(m[pt] + dz[:, 6:7]).clamp(*wl.opt.m_range), (mu[pt] + dz[:, 7:]).clamp(*wl.opt.mu_range)], 1).float(),
               shape=torch.as_tensor(wl.shape_id.astype(np.int32), device=dev), iters=torch.as_tensor(wl.iters.astype(np.int32), device=dev),
               q=torch.as_tensor(wl.q_traj, device=dev).contiguous())
    if pd:
        ten.update(qj=st["qj"][pt].float().contiguous(), qd=st["qd"][pt].float().contiguous())
    # the true environment's observations (the lead-in's settings), with sensor noise
    one = Reference(lead, [0], [8], dev)
    gt = {k: a[B:] for k, a in st.items()}
    T, P = case["frames"], wl.scene.n_pads
    obs, gone = [], torch.zeros(1, dtype=torch.bool, device=dev)
    oq, opp = [], []
    for f in range(F0, F0 + T):
        gt, fo, gone = one.frame(gt, m[B:], mu[B:], f, gone)
        obs.append(fo[0])
        if pd:
            oq.append(gt["qj"][0])
            lp, lq, _, _ = one.fk(gt["qj"])
            mid = [0.5 * (max(a, 0.0) + min(b, 1.0)) * one.len for a, b in zip(wl.scene.pad_s0, wl.scene.pad_s1)]
            opp.append(torch.stack([torch.cat([lp[0, l] + qmat(lq[0, l])[:, 0] * mid[k], torch.zeros(1, dtype=F64, device=dev), lq[0, l]])
                                    for k, l in enumerate(wl.scene.pad_link)]))
    ten["obs"] = (torch.stack(obs) + t(rng.normal(0, 0.002, (T, P, 3)))).float().contiguous()
    if pd:
        ang, slips = rng.uniform(0, 2 * math.pi, (T, P)), rng.random((T, P)) < 0.5
        bits = (slips + 2 * (rng.random((T, P)) < 0.3)).astype(np.int32)
        slip = np.stack([np.cos(ang) * slips, np.sin(ang) * slips, np.zeros((T, P)), np.zeros((T, P))], -1).astype(np.float32)
        slip[..., 2] = bits.view(np.float32)
        ten.update(obs_q=torch.stack(oq).float().contiguous(), obs_pp=torch.stack(opp).float().contiguous(),
                   obs_slip=torch.as_tensor(slip, device=dev).contiguous())
    if case.get("envs"):
        ten["envs"] = torch.as_tensor(np.sort(rng.choice(n, case["envs"], replace=False)).astype(np.int32), device=dev)
    return wl, ten


def prepare(case, seed):
    wl, ten = inputs(case, seed)
    sim = inhand.make_sim(wl, seed=seed)
    sim.sim_set_commands(0, ten["q"])
    sim.sim_set_state(ten["pose"], ten["vel"], ten["params"], ten["shape"], ten["iters"])
    dev = ten["pose"].device
    T = case["frames"]
    ten.update(est=torch.zeros(T, 8, device=dev), argmin=torch.zeros(T, dtype=torch.int32, device=dev),
               cost=torch.zeros(case["n"], dtype=F64, device=dev), parent=torch.zeros(case["n"], dtype=torch.int32, device=dev))
    return dict(case=case, wl=wl, sim=sim, **ten)


def run(state):
    s, sim, kind, T = state, state["sim"], state["case"]["kind"], state["case"]["frames"]
    if kind == "grad" and "envs" not in s:
        pose, params = s["pose"].detach().requires_grad_(), s["params"].detach().requires_grad_()
        cost = autograd.tracking_cost(sim, pose, params, s["vel"], F0, s["obs"])
        cost.sum().backward()
        return dict(cost=cost.detach(), pose_grad=pose.grad, params_grad=params.grad)
    sim.sim_set_state(s["pose"], s["vel"], s["params"])
    if kind == "grad":
        cost, grad, _ = sim.sim_adjoint(F0, s["obs"], envs=s["envs"])
        return dict(cost=cost, grad=grad)
    out = dict(est=s["est"], argmin=s["argmin"])
    if kind == "frames" and T == 1:
        sim.sim_step_track(F0, s["obs"][0], s["cost"], s["argmin"], s["est"][0])
    elif kind == "frames":
        sim.sim_step_frames(F0, s["obs"])
        sim.sim_frames_argmin(s["est"], s["argmin"])
    elif kind == "window":
        sim.sim_track_window(F0, s["obs"], s["wl"].opt, 0, s["est"], s["argmin"])
    elif kind == "calls":
        sim.sim_step(F0, 1)
        out["forces"], _ = sim.sim_read_sensors()
        sim.cost_eval(s["obs"][0], s["cost"], s["argmin"], s["est"][0])
        sim.optimizer_update(s["wl"].opt, 0, None, s["parent"])
        out.update(cost=s["cost"], parent=s["parent"])
    else:
        sim.sim_set_hand(s["qj"], s["qd"])
        sim.sim_step_frames_full(F0, s["obs_q"], s["obs_pp"], s["obs"], s["obs_slip"])
        sim.sim_frames_argmin(s["est"], s["argmin"])
        _, out["pad_pose"], out["slip"] = sim.sim_read_observation()
        out["q"], out["qd"] = sim.sim_get_hand()
    out["pose"], out["vel"], out["params"], out["status"] = sim.sim_get_state()
    if kind in ("frames", "pd"):
        out["forces"], _ = sim.sim_read_sensors()
    return out


def exact(case, seed):
    kind, T = case["kind"], case["frames"]
    if case.get("warm") or kind == "window":
        return None   # a cache or a resample between the frames: not one closed computation
    if kind == "grad" and case.get("envs", case["n"]) * T > 2048:
        return None   # too long on one card in FP64 with every iteration kept for the backward
    wl, ten = inputs(case, seed)
    dev = ten["pose"].device
    if kind == "grad":
        at = ten["envs"].long() if "envs" in ten else torch.arange(case["n"], device=dev)
        shape, iters = wl.shape_id[at.cpu().numpy()], wl.iters[at.cpu().numpy()]
        ref = Reference(wl, shape, iters, dev, smooth=(1e3, float(np.float32(1e-3))))
        x, q = (ten["pose"][at, a:b].to(F64).requires_grad_() for a, b in ((0, 3), (4, 8)))
        par = ten["params"][at].to(F64).requires_grad_()
        v8 = ten["vel"][at].to(F64)
        st = dict(x=x, q=q, v=v8[:, :3], w=v8[:, 4:7])
        dead = torch.zeros(len(at), dtype=torch.bool, device=dev)
        cost = torch.zeros(len(at), dtype=F64, device=dev)
        tau2 = float(np.float32(wl.sim.tau)) ** 2
        for k in range(T):
            st, fo, dead = ref.frame(st, par[:, :1], par[:, 1:], F0 + k, dead)
            o = ten["obs"][k].to(F64)
            cost = cost + wl.sim.w_force * ((fo - o) ** 2).sum((1, 2))
            cost = cost + wl.sim.w_contact * (((fo.detach() ** 2).sum(-1) > tau2) != ((o ** 2).sum(-1) > tau2)).sum(1)
        gx, gq, gp = torch.autograd.grad(cost.sum(), (x, q, par))
        if "envs" not in ten:
            return dict(cost=cost.detach(), pose_grad=pose8(gx, gq), params_grad=gp)
        turn = qmul(gq, q.detach() * torch.tensor([1.0, -1, -1, -1], dtype=F64, device=dev))[:, 1:] / 2
        return dict(cost=cost.detach(), grad=torch.cat([gx, turn, gp], 1))
    with torch.no_grad():
        st, m, mu = state_of(ten, kind == "pd")
        ref = Reference(wl, wl.shape_id, wl.iters, dev)
        dead = torch.zeros(case["n"], dtype=torch.bool, device=dev)
        for k in range(T):
            st, fo, dead = ref.frame(st, m, mu, F0 + k, dead)
        if kind == "calls":   # the resampled state has random draws in it; the stepped frame's forces do not
            return dict(forces=fo, est=None, argmin=None, cost=None, parent=None, pose=None, vel=None, params=None, status=None)
        out = dict(est=None, argmin=None, pose=pose8(st["x"], st["q"]), vel=vel8(st["v"], st["w"]), params=ten["params"].to(F64),
                   status=None, forces=fo)
        if kind == "pd":
            out.update(q=st["qj"], qd=st["qd"], pad_pose=None, slip=None)
        return out


def work(case):
    """State, forces and frame outputs read and written once; the contact, pair and iteration arithmetic of typical grasps."""
    spheres, contacts, tests, links, pads, ns, iters = {   # contacts and sphere tests of an environment's substep
        "tracking_box27": (27, 12, 200, 17, 8, 2, 20), "tracking_cyl64": (64, 80, 500, 17, 8, 2, 20),
        "uneven_mixed": (91, 30, 180, 21, 16, 2, 23), "sweep_mug128": (128, 58, 560, 21, 16, 4, 40)}[case["workload"]]
    iters = case.get("iters", iters)
    n, T = case.get("envs", case["n"]) if case["kind"] == "grad" else case["n"], case["frames"]
    flops = n * T * ns * (184 + 25 * links + 15 * spheres + 41 * tests + 91 * contacts + iters * (24 + 89 * contacts))
    byts = n * (152 + 12 * pads) + T * pads * 12 + T * 36
    if case["kind"] == "grad":
        flops, byts = 3 * flops, n * (72 + 56) + T * pads * 12   # forward, and a reverse of twice its work
    if case["kind"] == "pd":
        flops, byts = flops * 1.2, byts + n * (4 * 64 + 48 * pads)
    if case["kind"] in ("window", "calls"):
        byts += n * 72
    return {"bytes": byts, "flops": flops}
