"""The step's results depend neither on the lanes that execute an environment nor on
the warps that an SM holds: a batch large enough for two environments to a warp
(box), or for more warps to an SM with fewer registers (box, cylinder), against the
same environments in a small batch, bit for bit. The sums' order is fixed by the
shape's width alone, so the tolerance is zero."""
import dataclasses

import numpy as np
import pytest

from gpu_common import dev
from paper_2002_12160_gb300 import workloads as W

torch = pytest.importorskip("torch")


def _run(wl, n, shape, frames):
    from paper_2002_12160_gb300 import inhand
    sim = inhand.make_sim(wl, n_envs=n, max_frames=frames)
    sim.sim_set_commands(0, torch.from_numpy(wl.q_traj[:frames + 1]).contiguous().to(dev()))
    sim.sim_sample_initial(wl.nominal_pose, wl.init.sigma_p, wl.init.sigma_r, wl.init.m_range, wl.init.mu_range)
    its = torch.from_numpy(np.resize(np.array([20, 3, 0, 11], np.int32), n)).to(dev())   # neighbours of a warp stop at different counts
    pose, vel, par, _ = sim.sim_get_state()
    sim.sim_set_state(pose, vel, par, torch.zeros(n, dtype=torch.int32, device=dev()), its)
    sim.sim_set_variant(*shape)
    sim.sim_step(0, frames)
    out = [*sim.sim_get_state(), sim.sim_read_sensors()[0]]
    return [t.cpu() for t in out]


@pytest.mark.gpu
@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("name,shape", [("tracking_box27", (16, 2)), ("tracking_box27", (32, 2)), ("tracking_box27", (64, 2)),
                                        ("tracking_cyl64", (32, 2)), ("tracking_cyl64", (64, 2)), ("tracking_cyl64", (128, 1))])
def test_results_do_not_depend_on_the_lanes(name, shape, warm):
    n_big, n_small = 4097, 41   # odd: the last warp of two holds one environment
    wl = W.make_workload(name, n_envs=n_big, frames=20)
    wl.sim = dataclasses.replace(wl.sim, warm_start=warm)
    big, small = _run(wl, n_big, shape, 20), _run(wl, n_small, shape, 20)
    assert small[-1].abs().max() > 0.01   # the fingers carry force
    for a, b in zip(big, small):
        assert torch.equal(a[:n_small], b)
