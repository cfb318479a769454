"""The PD-driven hand at the edges of its register slots: substeps of up to 32, 64, 96
and 128 contacts (1 to 4 slots a lane) and beyond (memory), hands of up to 16 joints
(two lanes a joint) and of 20 (one), one frame against the oracle with the one-frame
parity's tolerances (test_gpu_pd.py)."""
import numpy as np
import pytest

import oracle as O

from gpu_common import scene32, sim32, start
from test_gpu_pd import _hand_state, _pd, compare_pd_frame

pytestmark = pytest.mark.gpu

# (workload, environments, lead-in frames, the slot counts its substeps reach: 5 = memory)
CASES = [("tracking_box27", 24, 11, {1}), ("tracking_cyl64", 96, 15, {3, 4}),
         ("uneven_mixed", 80, 9, {1, 2, 5}), ("sweep_mug128", 40, 9, {1, 2})]


@pytest.mark.parametrize("name,n,lead,slots", CASES)
def test_pd_frame_parity_over_the_slots(name, n, lead, slots):
    wl = _pd(name, n, lead + 2)
    sim = start(wl, n=n, frames=lead + 2)
    sim.sim_step(0, lead)
    st = _hand_state(sim, wl.shape_id[:n].astype(np.int32), wl.iters[:n].astype(np.int32))
    _, diag = O.step_pd(O.OracleScene(scene32(wl.scene)), sim32(wl.sim), st, wl.q_traj, lead, 1)
    per_substep = diag[:, 0] / wl.sim.substeps
    reached = {min(int(np.ceil(c / 32)), 5) for c in per_substep if c > 0}
    assert slots <= reached
    compare_pd_frame(wl, sim, lead)
