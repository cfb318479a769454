"""A tracking window after a longer window of frames has grown the buffers that its
captured graph writes: the same bits as on a handle that never took the longer one."""
import pytest

from gpu_common import dev, start, torch
from paper_2002_12160_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHORT, LONG = 3, 9


@pytest.mark.parametrize("n", [40, 3000])
def test_window_after_the_frame_buffers_grew(n):
    d = dev()
    wl = W.make_workload("tracking_box27", n_envs=n, frames=30)
    obs = torch.zeros((LONG, wl.scene.n_pads, 3), device=d)
    outs = []
    for grow in (False, True):
        sim = start(wl, n=n, frames=30)
        sim.sim_step(0, 12)
        pose, vel, params, _ = (t.clone() for t in sim.sim_get_state())
        est, best = torch.zeros((SHORT, 8), device=d), torch.zeros(SHORT, dtype=torch.int32, device=d)
        sim.sim_track_window(12, obs[:SHORT], wl.opt, 1, est, best)
        if grow:
            sim.sim_step_frames(12, obs)
            sim.sim_frames_argmin()
            sim.optimizer_update(wl.opt, 2)
        sim.sim_set_state(pose, vel, params)
        est2, best2 = torch.zeros_like(est), torch.zeros_like(best)
        sim.sim_track_window(12, obs[:SHORT], wl.opt, 3, est2, best2)
        outs.append([est, best, est2, best2, *sim.sim_get_state()])
        torch.cuda.synchronize()
        sim.close()
    assert all(torch.equal(a, b) for a, b in zip(*outs))
    assert outs[0][2].abs().sum() > 0
