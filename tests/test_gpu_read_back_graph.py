"""The read-backs inside a caller's captured graph, on the caller's own stream: each
replay copies the state of that moment, exactly."""
import pytest

from gpu_common import dev, start, torch
from paper_2002_12160_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_read_backs_replay_in_a_captured_graph():
    wl = W.make_workload("tracking_box27", n_envs=33, frames=12)
    sim = start(wl, n=33, frames=12)
    d = dev()
    forces, status = sim.sim_read_sensors()
    st = torch.cuda.Stream(d)
    st.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        sim.sim_read_sensors(forces, status)
        with torch.cuda.graph(g, stream=st):
            pose, vel, params, st2 = sim.sim_get_state()
            sim.sim_read_sensors(forces, status)
    torch.cuda.synchronize()
    for f in range(3):
        sim.sim_step(4 * f, 4)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        want = sim.sim_get_state()
        assert all(torch.equal(a, b) for a, b in zip((pose, vel, params, st2), want)), f
        wf, ws = sim.sim_read_sensors()
        assert torch.equal(forces, wf) and torch.equal(status, ws), f
    assert forces.abs().max() > 0
