"""Contacts beyond the 128 that a warp or a block keeps in registers and shared memory
(64 in the two-environment warps of the 16-wide shapes): 256-sphere composites around
one heavy grasp, with 150 to 210 contacts a substep. The step of every summation width,
cold and warm-started, is compared with the oracle's one-frame step, and the adjoint of
both warp counts with the FP64 adjoint, at the tolerances of the one-frame parity and of
the N = 4 adjoint tests. Each asserts that its environments do hold more contacts."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from oracle import adjoint as A
from paper_2002_12160_gb300 import workloads as W

from gpu_common import FRAGILE, assert_report, compare_frame, dev, oracle_state, scene32, sim32, start, torch

pytestmark = pytest.mark.gpu

N, LEAD, H = 24, 12, 2
MARGINS = [None, 0.003, 0.005]   # the workload's own, and two that add contacts
BLOCKS = [slice(0, 3), slice(3, 6), slice(6, 7), slice(7, 8)]


def _heavy(margin, warm=False):
    """N copies of the sampled grasp with the most contacts, positions and parameters spread."""
    wl = W.make_workload("uneven_mixed", n_envs=64, frames=LEAD + H + 4)
    wl.shape_id[:] = 3   # the composite of 256 spheres
    if margin:
        wl.sim = dataclasses.replace(wl.sim, margin=margin)
    wl.sim = dataclasses.replace(wl.sim, warm_start=warm)
    sim = start(wl, n=64, frames=LEAD + H + 4)
    sim.sim_step(0, LEAD)
    state = sim.sim_get_state()
    probe = oracle_state(state, wl.shape_id[:64].astype(np.int32), wl.iters[:64].astype(np.int32))
    osc, sm = O.OracleScene(scene32(wl.scene)), dataclasses.replace(sim32(wl.sim), warm_start=False)
    _, diag = O.step(osc, sm, probe, wl.q_traj, LEAD, 1)
    heavy = int(np.where(probe.status == 0, diag[:, 0], -1).argmax())
    sim.close()
    r = np.random.default_rng(11)
    wl.shape_id, wl.iters = wl.shape_id[:N], wl.iters[:N]
    sim = start(wl, n=N, frames=LEAD + H + 4)
    pose, vel = (t[heavy:heavy + 1].repeat(N, 1) for t in state[:2])
    pose[:, :3] += torch.from_numpy(r.normal(0.0, 2e-4, (N, 3)).astype(np.float32)).to(dev())
    params = torch.from_numpy(np.stack([r.uniform(0.05, 0.3, N), r.uniform(0.3, 1.2, N)], 1).astype(np.float32)).to(dev())
    sim.sim_set_state(pose.contiguous(), vel.contiguous(), params,
                      *(torch.from_numpy(a.astype(np.int32)).to(dev()) for a in (wl.shape_id, wl.iters)))
    return wl, sim


@pytest.mark.parametrize("margin", MARGINS)
@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("shape", [(16, 2), (32, 2), (64, 2), (128, 1)])
def test_step_with_many_contacts_matches_oracle(shape, warm, margin):
    wl, sim = _heavy(margin, warm)
    sim.sim_set_variant(*shape)
    for frame in range(LEAD, LEAD + 2):   # (the second frame of a warm-started handle starts from cached impulses)
        rep = compare_frame(wl, sim, frame)
        ok = rep["ok"] & (rep["status_or"] == 0)
        assert ok.sum() >= N // 2 and rep["diag"][ok, 0].min() > 128 * wl.sim.substeps
        assert_report(rep, min_ok_frac=0.5)
    sim.close()


@pytest.mark.parametrize("margin", MARGINS)
def test_adjoint_with_many_contacts_matches_oracle(margin):
    wl, sim = _heavy(margin)
    shape, iters = wl.shape_id.astype(np.int32), wl.iters.astype(np.int32)
    st = oracle_state(sim.sim_get_state(), shape, iters)
    sc, sm = scene32(wl.scene), sim32(wl.sim)
    osc = O.OracleScene(sc)
    probe = O.State(st.pose, st.vel, st.theta, shape, iters)
    truth = O.State(st.pose[:1], st.vel[:1], np.array([wl.theta_gt], np.float64), shape[:1], iters[:1])
    obs, fragile, fewest = [], np.zeros(N, bool), np.full(N, np.inf)
    for k in range(H):
        f, _ = O.step(osc, sm, truth, wl.q_traj, LEAD + k, 1)
        obs.append(f[0])
        _, diag = O.step(osc, sm, probe, wl.q_traj, LEAD + k, 1)
        fragile |= (diag[:, 2] < FRAGILE) | (diag[:, 3] < FRAGILE) | (diag[:, 4] < FRAGILE)
        fewest = np.minimum(fewest, diag[:, 0] / wl.sim.substeps)
    obs = np.asarray(obs, np.float32)
    picked = np.nonzero(~fragile & (probe.status == 0) & (fewest > 128))[0]
    assert len(picked) >= 6, (fragile.sum(), fewest)
    want = {i: A.horizon(sc, sm, st.pose[i], st.vel[i], st.theta[i], wl.q_traj, LEAD, H, obs.astype(np.float64), shape=3,
                         iters=int(iters[i]))[:2] for i in picked}
    o = torch.from_numpy(obs).to(dev())
    for variant in [(4, 1), (1, 1)]:
        sim.sim_set_adjoint_variant(*variant)
        cost, grad, _ = sim.sim_adjoint(LEAD, o, checkpoint_every=1)
        cost, grad = cost.cpu().numpy(), grad.cpu().numpy().astype(np.float64)
        for i, (c_or, g_or) in want.items():
            assert abs(cost[i] - c_or) <= 1e-3 * abs(c_or) + 1e-6, (variant, i, cost[i], c_or)
            floor = 1e-3 * max(np.linalg.norm(g_or[b]) for b in BLOCKS)
            for b in BLOCKS:
                err = np.linalg.norm(grad[i, b] - g_or[b])
                assert err <= 1e-3 * np.linalg.norm(g_or[b]) + floor, (variant, i, b, grad[i, b], g_or[b])
    sim.close()


@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("shape", [(32, 2), (64, 2), (128, 1)])
def test_large_batches_step_many_contacts_to_the_same_bits(shape, warm):
    """Few environments update the first contact past a lane's slots beside them, many do
    not (at most two rounds of twelve one-warp blocks an SM do)."""
    wl, sim = _heavy(0.005, warm)
    pose, vel, params, _ = (t.clone() for t in sim.sim_get_state())
    shape_id, iters = (torch.from_numpy(a.astype(np.int32)).to(dev()) for a in (wl.shape_id, wl.iters))
    sms = torch.cuda.get_device_properties(dev()).multi_processor_count
    copies = 2 * 12 * sms // N + 1
    wl.shape_id, wl.iters = np.tile(wl.shape_id, copies), np.tile(wl.iters, copies)
    big = start(wl, n=N * copies, frames=LEAD + H + 4)
    for handle, k in ((sim, 1), (big, copies)):
        handle.sim_set_variant(*shape)
        handle.sim_set_state(*(t.repeat(k, *[1] * (t.dim() - 1)).contiguous() for t in (pose, vel, params, shape_id, iters)))
        handle.sim_step(LEAD, 3)
    want = [*sim.sim_get_state(), *sim.sim_read_sensors()]
    for a, b in zip(want, [*big.sim_get_state(), *big.sim_read_sensors()]):
        assert torch.equal(a, b[:N]) and torch.equal(a, b[-N:])
    assert not want[3].any()
    big.close()
    sim.close()


def test_four_warps_agree_with_and_without_a_second_contact_a_thread():
    """The four-warp kernels for scenes of up to 128 contacts and of more, on environments
    that either can hold (the contact capacity is all that differs)."""
    n, res = 40, []
    for c_max in (128, 256):
        wl = W.make_workload("tracking_cyl64", n_envs=n, frames=LEAD + 6)
        wl.sim = dataclasses.replace(wl.sim, c_max=c_max)
        sim = start(wl, n=n, frames=LEAD + 6)
        sim.sim_step(0, LEAD)
        sim.sim_set_adjoint_variant(4, 1)
        obs = torch.zeros((4, wl.scene.n_pads, 3), dtype=torch.float32, device=dev())
        res.append(sim.sim_adjoint(LEAD, obs, checkpoint_every=2, want_quat=True))
        assert not sim.sim_get_state()[3].any()
        sim.close()
    assert all(torch.equal(a, b) for a, b in zip(*res)) and torch.isfinite(res[0][1]).all()
