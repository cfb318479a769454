"""The elite update at the edges of its draws' blocks (one warp of eight environments up
to 4096 of them, four warps beyond): every parent exactly, and the states, as the
one-size test of the update against the oracle."""
import pytest

import test_gpu_parity as parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 9, 4096, 4097])
def test_update_matches_oracle_at_the_block_edges(n):
    parity.test_optimizer_update_matches_oracle(n)
