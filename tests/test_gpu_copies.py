"""State, sensors and joints are read back (and the joints set) by one launch over all
arrays: the same values into aligned arrays, into arrays at odd 4-byte offsets, in
parts, and into pinned host memory (copied by calls), exactly."""
import dataclasses

import pytest

from gpu_common import dev, start, torch
from paper_2002_12160_gb300 import inhand
from paper_2002_12160_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 300])
def test_read_back_into_any_arrays(n):
    wl = W.make_workload("tracking_cyl64", n_envs=n, frames=6)
    wl.sim = dataclasses.replace(wl.sim, hand="pd")
    sim = start(wl, n=n, frames=6)
    sim.sim_step(0, 5)
    d, L, h = dev(), inhand.lib(), sim._h
    forces, status = sim.sim_read_sensors()
    q, pp, slip = sim.sim_read_observation()
    pose, vel, par, st = sim.sim_get_state()
    assert forces.abs().max() > 0 and torch.equal(st, status)
    # odd offsets
    f1 = torch.zeros(forces.numel() + 1, device=d)[1:].view_as(forces)
    s1 = torch.zeros(n + 3, dtype=torch.int32, device=d)[3:]
    sim.sim_read_sensors(f1, s1)
    assert torch.equal(f1, forces) and torch.equal(s1, status)
    q1 = torch.zeros(q.numel() + 3, device=d)[3:].view_as(q)
    sim.sim_read_observation(q1, torch.empty_like(pp), torch.empty_like(slip))
    assert torch.equal(q1, q)
    # one array alone, and pinned host memory
    p1, v1 = torch.zeros_like(pose), torch.zeros_like(vel)
    assert L.sim_get_state(h, p1.data_ptr(), None, None, None) == 0
    assert torch.equal(p1, pose)
    hp, hv, ht, hs = (torch.zeros(t.shape, dtype=t.dtype, pin_memory=True) for t in (pose, vel, par, st))
    assert L.sim_get_state(h, hp.data_ptr(), v1.data_ptr(), ht.data_ptr(), hs.data_ptr()) == 0
    sim.sim_sync()
    assert torch.equal(hp, pose.cpu()) and torch.equal(v1, vel) and torch.equal(ht, par.cpu()) and torch.equal(hs, st.cpu())
    # the joints in, from odd offsets
    qn = torch.arange(q.numel() + 1, dtype=torch.float32, device=d)[1:].view_as(q) * 1e-3
    qdn = torch.flip(qn, (0, 1)).contiguous()
    sim.sim_set_hand(qn, qdn)
    a, b = sim.sim_get_hand()
    assert torch.equal(a, qn) and torch.equal(b, qdn)
    sim.sim_set_hand(qn)
    a, b = sim.sim_get_hand()
    assert torch.equal(a, qn) and not b.any()
