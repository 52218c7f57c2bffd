"""Lists of one trial of every size class of the list build (four, two or one
warp per cluster), against the FP64 oracle's pair set."""
import numpy as np
import pytest

import oracle as O
from paper_1405_6104_gb300 import binding as B
from paper_1405_6104_gb300 import systems as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1405_6104_gb300 import build
    build.build()
    B.load()


@pytest.mark.parametrize("n_water", [430, 1500, 1700, 2100, 2800, 3500, 4200])
def test_pairs_are_the_oracles(n_water):
    """The oracle takes a pair by atom index, the kernels by cluster order, and
    the image of one atom or the other rounds: pairs within that rounding of
    the list radius (each component of the difference off by an ulp of a
    coordinate, the squares' sum by three) may belong to one set only."""
    s, p = S.small_solvated(n_solute=24, n_water=n_water)
    with B.TrialBatch(s, p, [1], trial_seeds=[3]) as b:
        b.step(7)
        pos = B.sim_list_positions(b.h, 0)
        got = B.sim_pairlist(b.h, 0)
    r_list = p.r_cut + p.skin
    ref = O.pairlist(s, pos.astype(np.float32), r_list)
    got, ref = ({tuple(x) for x in q.tolist()} for q in (got, ref))
    assert len(ref) > 50 * s.n_atoms
    box = float(np.float32(s.box))
    for i, j in got ^ ref:
        d = pos[j] - pos[i]
        r = np.linalg.norm(d - box * np.round(d / box))
        assert abs(r - r_list) <= 2.0 ** -23 * (np.sqrt(3.0) * box + 3.0 * r_list), (i, j, r)
    assert len(got ^ ref) <= 4
