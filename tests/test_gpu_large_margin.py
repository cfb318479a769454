"""Margins far above any distance: every (link, sphere) pair is a contact, and nothing
else is -- the places that fill a shape's last cluster of eight stay empty -- so every
such margin gives the bits of a margin of one metre: the step, the PD-driven hand and
the adjoint, for shapes that end 1, 2 and 7 spheres into a cluster."""
import dataclasses

import numpy as np
import pytest

from gpu_common import dev, start, torch
from paper_2002_12160_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spheres", [7, 9, 10])
@pytest.mark.parametrize("hand", ["kinematic", "pd"])
def test_large_margins_add_no_contacts(spheres, hand):
    n, d, ref = 5, dev(), None
    for margin in (1.0, 1e15, 1e18, 3e18, 1e19, 1e20, float("inf")):
        wl = W.make_workload("tracking_box27", n_envs=n, frames=8)
        wl.scene.shapes = [np.ascontiguousarray(wl.scene.shapes[0][:spheres])]
        wl.sim = dataclasses.replace(wl.sim, margin=margin, hand=hand, c_max=256)
        sim = start(wl, n=n, frames=8)
        sim.sim_work_counters(reset=True)
        sim.sim_step(0, 2)
        w = sim.sim_work_counters()
        assert w["contacts"] == w["env_substeps"] * spheres * wl.scene.n_links, margin
        out = [*sim.sim_get_state(), *sim.sim_read_sensors()]
        if hand == "kinematic":
            obs = torch.zeros((2, wl.scene.n_pads, 3), device=d)
            for shape in ((4, 1), (1, 1)):
                sim.sim_set_adjoint_variant(*shape)
                out += list(sim.sim_adjoint(2, obs, want_quat=True))
        assert not out[3].any()
        ref = ref or out
        assert all(torch.equal(a, b) for a, b in zip(ref, out)), margin
