"""The REPS temperature where a few costs lie far above the rest: the root of the dual
is then any distance below the costs' range, down to e^-180 of it here, and every
parent is still the one that the FP64 oracle draws."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from gpu_common import dev, oracle_state, start
from paper_2002_12160_gb300 import workloads as W

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("n", [64, 700])
@pytest.mark.parametrize("w_force,w_contact", [(1.0, 1e20), (1e-10, 1e35), (1e-30, 1e38), (1e-38, 1e38)])
def test_reps_parents_with_outlying_costs(n, w_force, w_contact):
    wl = W.make_workload("tracking_box27", n_envs=n, frames=20)
    wl.sim = dataclasses.replace(wl.sim, w_force=w_force, w_contact=w_contact)
    sim = start(wl, n=n, frames=20)
    d = dev()
    sim.sim_step(0, 17)
    # one grasp with masses spread by up to 10 %, whose costs differ by the forces alone;
    # every eighth object out of reach, whose contact states are all wrong
    pose, vel, params, _ = (t.clone() for t in sim.sim_get_state())
    forces, _ = sim.sim_read_sensors()
    e = int(forces.norm(dim=(1, 2)).argmax())
    pose[:], vel[:], params[:] = pose[e].clone(), vel[e].clone(), params[e].clone()
    params[:, 0] *= torch.linspace(0.9, 1.1, n, device=d)
    pose[::8, 2] += 0.2
    sim.sim_set_state(pose, vel, params)
    sim.sim_step(17, 1)
    forces, _ = sim.sim_read_sensors()
    cm = torch.empty(n, dtype=torch.float64, device=d)
    sim.cost_eval(forces[n // 2 + 1].clone(), cm)
    costs = cm.cpu().numpy()
    far = costs >= 0.5 * w_contact
    assert np.isfinite(costs).all() and n // 8 <= far.sum() <= n // 2 and (costs[~far] > 0).sum() > n // 4
    before = oracle_state(sim.sim_get_state())
    eps = float(np.float32(0.5 * np.log(n)))
    opt = dataclasses.replace(wl.opt, kind="reps", reps_epsilon=eps)
    am = torch.empty(1, dtype=torch.int32, device=d)
    par = torch.empty(n, dtype=torch.int32, device=d)
    sim.optimizer_update(opt, 4, am, par)
    istar, parent, _ = O.softmax_update(opt, before, costs, wl.seed, 4)
    assert int(am.item()) == istar
    np.testing.assert_array_equal(par.cpu().numpy(), parent)
    assert len(set(parent.tolist())) > 1
