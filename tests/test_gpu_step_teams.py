"""Small batches of the 128-wide sums run a team of four warps an environment, larger ones
one warp: the same environments, copied until the device holds no team for each, give
the same bits everywhere -- states, forces, costs, window means, estimates, impulse
caches -- and the work counters are the copies' multiple."""
import dataclasses

import numpy as np
import pytest

from gpu_common import dev, start, torch
from paper_2002_12160_gb300 import workloads as W

pytestmark = pytest.mark.gpu
LEAD, N = 14, 37


def _outputs(sim, state, copies, obs, warm):
    sim.sim_set_variant(128, 1)
    sim.sim_set_state(*(t.repeat(copies, *[1] * (t.dim() - 1)).contiguous() for t in state))
    sim.sim_work_counters(reset=True)
    d, n = dev(), N * copies
    cost = [torch.empty(n, dtype=torch.float64, device=d) for _ in range(2)]
    arg = [torch.empty(k, dtype=torch.int32, device=d) for k in (1, 1, 3)]
    est = [torch.empty(8, dtype=torch.float32, device=d) for _ in range(2)] + [torch.empty((3, 8), dtype=torch.float32, device=d)]
    for k in range(2):   # scored frames, one a launch
        sim.sim_step_track(LEAD + k, obs[k], cost[k], arg[k], est[k])
    sim.sim_step_frames(LEAD + 2, obs[2:].contiguous())   # ... and three a launch
    sim.sim_frames_argmin(est[2], arg[2])
    sim.sim_step(LEAD + 5, 2)
    per_env = [*sim.sim_get_state(), *sim.sim_read_sensors(), *cost]
    if warm:
        count, lam, pair = sim.sim_get_warm_cache()
        held = torch.arange(pair.shape[1], device=d) < count[:, None]
        per_env += [count, torch.where(held[..., None], lam, 0.0), torch.where(held, pair, 0)]
    work = sim.sim_work_counters()
    return per_env, arg + est, work


@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("name", ["tracking_box27", "tracking_cyl64", "sweep_mug128", "uneven_mixed"])
def test_teams_give_the_bits_of_one_warp(name, warm):
    sms = torch.cuda.get_device_properties(dev()).multi_processor_count
    copies = 3 * sms // N + 1
    wl = W.make_workload(name, n_envs=N, frames=LEAD + 10)
    wl.sim = dataclasses.replace(wl.sim, warm_start=warm)
    sim = start(wl, n=N, frames=LEAD + 10)
    sim.sim_step(0, LEAD)
    pose, vel, params, _ = (t.clone() for t in sim.sim_get_state())
    params[5, 0] = -1.0   # an invalid environment, and one without iterations
    iters = np.asarray(wl.iters[:N], np.int32).copy()
    iters[7] = 0
    wl.shape_id = np.asarray(wl.shape_id[:N])
    state = (pose, vel, params, *(torch.from_numpy(np.asarray(a, np.int32)).to(dev()) for a in (wl.shape_id, iters)))
    forces = sim.sim_read_sensors()[0]
    obs = forces[:1].repeat(5, 1, 1) * torch.linspace(0.5, 1.5, 5, device=dev())[:, None, None]
    wl.shape_id, wl.iters = np.tile(wl.shape_id, copies), np.tile(iters, copies)
    big = start(wl, n=N * copies, frames=LEAD + 10)
    few, few_best, few_work = _outputs(sim, state, 1, obs, warm)
    many, many_best, many_work = _outputs(big, state, copies, obs, warm)
    assert few[4].abs().max() > 0.01 and few[3][5] != 0
    for a, b in zip(few, many):
        assert torch.equal(a, b[:N]) and torch.equal(a, b[-N:])
    for a, b in zip(few_best, many_best):   # (the lowest index of equal costs is in the first copy)
        assert torch.equal(a, b)
    assert {k: v * copies for k, v in few_work.items()} == many_work
    sim.close()
    big.close()
