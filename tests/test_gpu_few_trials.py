"""Kernels that a batch too small to fill the GPU takes, at the sizes where
they can go wrong, against the one-kernel step (whose warps each take a whole
reaction-coordinate tile, pair list or list build): the states must agree bit
for bit."""
import numpy as np
import pytest

from paper_1405_6104_gb300 import binding as B
from paper_1405_6104_gb300 import systems as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1405_6104_gb300 import build
    build.build()
    B.load()


def _states(s, p, mode, trials=1, steps=(13, 10)):
    with B.TrialBatch(s, p, [trials], trial_seeds=list(range(21, 21 + trials))) as b:
        B.sim_set_step_mode(b.h, mode)
        for n in steps:
            b.step(n)
        return [b.get_state(t) for t in range(trials)]


@pytest.mark.parametrize("n_solute", [6, 31, 32, 33, 64, 65, 97])
def test_tiles_by_a_block_match_tiles_by_a_warp(n_solute):
    """Tile edges of the 32 x 32 contact-pair tiles: one partial tile, exact
    ones, one atom into the next; every pair near (a short chain) and few."""
    s, p = S.small_solvated(n_solute=n_solute, n_water=430 + n_solute)
    for x, y in zip(_states(s, p, 0), _states(s, p, 1)):
        assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1]) and np.array_equal(x[2], y[2])
