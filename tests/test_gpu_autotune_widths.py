"""The autotuner times each summation width once: shapes of one width report the same
time, and the shape chosen is the fastest width's first."""
import pytest

from gpu_common import start
from paper_2002_12160_gb300 import inhand
from paper_2002_12160_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_shapes_of_one_width_share_a_time():
    sim = start(W.make_workload("tracking_cyl64", n_envs=300, frames=8), n=300, frames=8)
    sim.sim_step(0, 4)
    chosen, ms = sim.sim_autotune(4, 2)
    first = {}
    for shape in inhand.step_variants():
        first.setdefault(shape[0], shape)
        assert ms[shape] > 0 and ms[shape] == ms[first[shape[0]]]
    assert chosen == min(first.values(), key=lambda s: ms[s])
    sim.close()
