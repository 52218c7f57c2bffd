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


@pytest.mark.parametrize("per_atom", [4, 5, 9, 16])
def test_lists_with_many_excluded_partners_are_bit_exact(per_atom):
    """Exclusion rows at the edges of the list build's passes (four partners
    per atom at a time), in the smallest box the system takes (half lists with
    pairs on both sides of it, pair-by-pair images): the oracle's pair set."""
    import oracle as O

    s, p = S.small_solvated(n_solute=24, n_water=420)
    rng = np.random.default_rng(per_atom)
    have = {i: set() for i in range(s.n_atoms)}
    for a, b in np.asarray(s.bonds):
        have[a].add(int(b)), have[b].add(int(a))
    for a, _, c in np.asarray(s.angles):
        have[a].add(int(c)), have[c].add(int(a))
    extra = []
    for i in range(0, s.n_atoms, 3):
        for j in rng.permutation(s.n_atoms)[:200]:
            j = int(j)
            if j != i and j not in have[i] and len(have[i]) < per_atom and len(have[j]) < per_atom:
                have[i].add(j), have[j].add(i)
                extra.append((i, j))
    s = s.copy()
    s.excl_pairs = np.array(extra, np.int32)
    assert max(len(v) for v in have.values()) == per_atom
    with B.TrialBatch(s, p, [1], trial_seeds=[3]) as b:
        b.step(7)
        pos = B.sim_list_positions(b.h, 0)
        got = {tuple(x) for x in B.sim_pairlist(b.h, 0).tolist()}
    ref = {tuple(x) for x in O.pairlist(s, pos.astype(np.float32), p.r_cut + p.skin).tolist()}
    assert got == ref and len(ref) > 10 * s.n_atoms


@pytest.mark.parametrize("crowd", [60, 127, 128, 129, 257, 512, 900])
def test_crowded_columns_give_the_oracles_pairs(crowd):
    """A grid column that holds about `crowd` atoms (below, at and beyond the
    threads that sort it, up to its capacity of 1024), several of them at the
    same height: the oracle's pair set, with the columns around nearly empty."""
    import oracle as O

    s, p = S.small_solvated(n_solute=24, n_water=432)
    rng = np.random.default_rng(crowd)
    pos = s.pos % s.box
    who = rng.permutation(s.n_atoms)[:crowd]
    pos[who, :2] = 0.5 * s.box + 0.02 * rng.random((crowd, 2))
    pos[who, 2] = np.round(rng.random(crowd) * s.box, 2)
    pos = pos.astype(np.float32).astype(np.float64)
    with B.TrialBatch(s, p, [1], trial_seeds=[3]) as b:
        b.set_state(0, pos, np.zeros_like(pos))
        at = B.sim_list_positions(b.h, 0)
        got = B.sim_pairlist(b.h, 0).tolist()
    ref = {tuple(x) for x in O.pairlist(s, at.astype(np.float32), p.r_cut + p.skin).tolist()}
    assert len(got) == len(ref) and {tuple(x) for x in got} == ref


def _lists(systems, p, mode):
    with B.TrialBatch(systems, p, [1] * len(systems), trial_seeds=list(range(3, 3 + len(systems)))) as b:
        B.sim_set_step_mode(b.h, mode)
        b.step(7)
        pairs = [B.sim_pairlist(b.h, k).astype(np.int64) for k in range(len(systems))]  # in no fixed order
        return [np.sort(x[:, 0] << 32 | x[:, 1]) for x in pairs], [b.get_state(k)[0] for k in range(len(systems))]


@pytest.mark.parametrize("n_water", [420, 1700, 2100, 3500, 4200])
def test_lists_shared_by_warps_match_lists_by_a_warp(n_water):
    """One trial's lists, each built by four warps (a few hundred clusters), by
    two, or by one: the one-kernel step's pairs, and its positions (the forces'
    sums follow the lists' order)."""
    s, p = S.small_solvated(n_solute=24, n_water=n_water)
    x, y = _lists([s], p, 0), _lists([s], p, 1)
    assert np.array_equal(x[0][0], y[0][0]) and np.array_equal(x[1][0], y[1][0])


@pytest.mark.parametrize("n_water", [3900, 4400, 8300])
def test_lists_of_trials_beyond_one_pass_of_the_binning(n_water):
    """A trial of about as many atoms as the binning's threads take in one pass
    (12 288), and in two and three, beside a small trial: the one-kernel step's
    pairs and positions, after rebuilds that start from a list's order."""
    big, p = S.small_solvated(n_solute=24, n_water=n_water)
    small, _ = S.small_solvated(n_solute=24, n_water=432)
    for x, y in zip(_lists([big, small], p, 0), _lists([big, small], p, 1)):
        assert all(np.array_equal(u, v) for u, v in zip(x, y))


@pytest.mark.parametrize("n_solute,n_water", [(6, 430), (37, 420), (60, 440)])
def test_one_pass_energies_match_the_general_kernel(n_solute, n_water):
    """Energies of the one-pass force and energy kernel (device tensors) and
    of the general energy kernel (energy_forces) on the same configuration and
    lists, bonds and angles strained, in the smallest boxes (pair-by-pair
    images): equal to the last bit of the fixed-point sums."""
    import torch

    from paper_1405_6104_gb300 import autograd as U

    s, p = S.small_solvated(n_solute=n_solute, n_water=n_water)
    rng = np.random.default_rng(n_solute)
    ev = U.Evaluator(s, p, n_conf=2)
    try:
        for k in range(3):  # the lists of the first serve the second, the third needs new ones
            x = s.pos[None] + 0.004 * rng.normal(size=(2, s.n_atoms, 3)) + (0.3 if k == 2 else 0.0)
            x = x.astype(np.float32).astype(np.float64)
            u, f = ev.device_energy_and_forces(torch.tensor(x, device="cuda"))
            for t in range(2):
                e, _ = ev.batch.energy_forces(t)
                assert float(u[t]) == pytest.approx(e[:4].sum(), rel=1e-15)
    finally:
        ev.close()
