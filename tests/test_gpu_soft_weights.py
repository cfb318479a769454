"""The WRS / REPS weights at the edges of the cluster's shares: sizes around
whole and partial chunks, CTAs without environments, all costs equal, one finite
cost; every parent and i* exactly as the FP64 oracle draws them."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from gpu_common import dev, oracle_state, start
from paper_2002_12160_gb300 import workloads as W

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 2, 511, 513, 4095, 4097])
@pytest.mark.parametrize("kind,temperature", [("reps", 0.25), ("reps", 0.999), ("wrs", 0.5)])
def test_weights_at_the_cluster_edges_match_oracle(n, kind, temperature):
    wl = W.make_workload("tracking_box27", n_envs=n, frames=20)
    sim = start(wl, n=n, frames=20)
    d = dev()
    sim.sim_step(0, 17)
    forces, _ = sim.sim_read_sensors()
    obs = forces[0].clone()
    for case in ("grasp", "one finite") if n > 2 else ("grasp",):
        if case == "one finite":   # every environment but the last made invalid
            pose, vel, params, _ = sim.sim_get_state()
            params = params.clone()
            params[:-1, 0] = -1.0
            sim.sim_set_state(pose, vel, params)
        cm = torch.empty(n, dtype=torch.float64, device=d)
        sim.sim_step(17, 1)
        sim.cost_eval(obs, cm)
        before = oracle_state(sim.sim_get_state())
        # REPS: a share of the bound at which all mass sits on the minima; WRS: the temperature itself
        t = float(np.float32(temperature * (np.log(max(n, 2)) if kind == "reps" else 1.0)))
        opt = dataclasses.replace(wl.opt, kind=kind, wrs_lambda=t, reps_epsilon=t)
        am = torch.empty(1, dtype=torch.int32, device=d)
        par = torch.empty(n, dtype=torch.int32, device=d)
        sim.optimizer_update(opt, 4, am, par)
        istar, parent, _ = O.softmax_update(opt, before, cm.cpu().numpy(), wl.seed, 4)
        assert int(am.item()) == istar
        np.testing.assert_array_equal(par.cpu().numpy(), parent)
