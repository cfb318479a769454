"""The adjoint at the edges of its register slots and of its tape's memory.

One warp per environment holds 32, 64, 96 or 128 contacts in 1 to 4 slots a lane and
the rest in memory; four warps hold one contact a thread, on as many warps as carry
contacts. Both are within 1e-3 per block (with an absolute floor of 1e-3 of the
environment's largest block) of the same exact gradient, so they are within twice
that of each other. A tape kept whole, by segments or by substeps gives the same bits."""
import numpy as np
import pytest

import oracle as O
from paper_2002_12160_gb300 import workloads as W

from gpu_common import FRAGILE, dev, oracle_state, scene32, sim32, start, torch

pytestmark = pytest.mark.gpu

BLOCKS = [slice(0, 3), slice(3, 6), slice(6, 7), slice(7, 8)]


def _started(n, warm, frames):
    wl = W.make_workload("uneven_mixed", n_envs=n, frames=frames)
    sim = start(wl, n=n, frames=frames)
    sim.sim_step(0, warm)
    return wl, sim


def test_slot_counts_agree_between_warp_counts():
    n, warm, H = 96, 12, 2
    wl, sim = _started(n, warm, warm + H + 2)
    st = oracle_state(sim.sim_get_state())
    probe = O.State(st.pose, st.vel, st.theta, wl.shape_id[:n].astype(np.int32), wl.iters[:n].astype(np.int32))
    osc, sm = O.OracleScene(scene32(wl.scene)), sim32(wl.sim)
    fragile, most = np.zeros(n, bool), np.zeros(n)
    for k in range(H):
        _, diag = O.step(osc, sm, probe, wl.q_traj, warm + k, 1)
        fragile |= (diag[:, 2] < FRAGILE) | (diag[:, 3] < FRAGILE) | (diag[:, 4] < FRAGILE)
        most = np.maximum(most, diag[:, 0] / wl.sim.substeps)   # contacts of a substep
    obs = torch.zeros((H, wl.scene.n_pads, 3), dtype=torch.float32, device=dev())
    res = []
    for shape in [(4, 1), (1, 1)]:
        sim.sim_set_adjoint_variant(*shape)
        c, g, _ = sim.sim_adjoint(warm, obs)
        res.append((c.cpu().numpy(), g.cpu().numpy().astype(np.float64)))
    (c4, g4), (c1, g1) = res
    classes = set()
    for i in range(n):
        if fragile[i] or not np.isfinite(c4[i]):
            continue
        assert abs(c1[i] - c4[i]) <= 2e-3 * abs(c4[i]) + 2e-6, (i, most[i], c1[i], c4[i])
        floor = 1e-3 * max(np.linalg.norm(g4[i, b]) for b in BLOCKS)
        for b in BLOCKS:
            assert np.linalg.norm(g1[i, b] - g4[i, b]) <= 2e-3 * np.linalg.norm(g4[i, b]) + 2 * floor, (i, most[i], b)
        if c4[i] > 0:
            classes.add(min(int(np.ceil(most[i] / 32)), 5))
    assert len(classes) >= 4, classes   # one to four slots, or memory


@pytest.mark.parametrize("shape", [(4, 1), (1, 1)])
def test_tape_memory_does_not_change_the_results(shape):
    n, warm, H = 8, 12, 6
    wl, sim = _started(n, warm, warm + H + 1)
    sim.sim_set_adjoint_variant(*shape)
    obs = torch.zeros((H, wl.scene.n_pads, 3), dtype=torch.float32, device=dev())
    ref = None
    # from a substep at a time (none fits) over every number of segments to the whole horizon
    for budget in [0, *(n * 250_000 * k for k in range(1, 16)), 16 << 30]:
        sim.sim_set_adjoint_memory(budget)
        for K in (1, 4):
            c, g, q = sim.sim_adjoint(warm, obs, checkpoint_every=K, want_quat=True)
            ref = ref or (c, g, q)
            assert all(torch.equal(a, b) for a, b in zip(ref, (c, g, q))), (budget, K)
