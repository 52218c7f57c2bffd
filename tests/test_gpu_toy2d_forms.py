"""The toy model's kernels in all their forms -- two lanes or one per trial,
prepared normals or tables, several launches -- and at parameters where a
divisor leaves the range their quotients are formed in: a trial is the same
bit for bit alone and among any number of others, and follows the oracle."""
import dataclasses

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


@pytest.mark.parametrize("bias", [S.TOY_NONE, S.TOY_RATCHET, S.TOY_STEERED])
@pytest.mark.parametrize("n,n_steps", [(17, 9000), (5000, 7000), (30000, 1500), (140000, 300)])
def test_trials_do_not_depend_on_their_number(n, n_steps, bias):
    """Pairs of lanes (few trials) against a lane each (many), normals
    prepared per launch against tables (from 2^25 draws on)."""
    tp = dataclasses.replace(S.Toy2dParams(), bias=bias)
    rng = np.random.default_rng(n)
    ks, seeds = rng.choice([0.5, 4.0, 16.0], n), rng.integers(1, 2 ** 60, n).astype(np.uint64)
    passage, phi, state, _ = B.toy2d_run(tp, ks, seeds, n_steps)
    sample = np.unique(np.concatenate([[0, 1, 15, 16, n - 1], rng.integers(0, n, 8)]))
    p1, f1, s1, path = B.toy2d_run(tp, ks[sample], seeds[sample], n_steps, path_every=7)
    assert np.array_equal(p1, passage[sample]) and np.array_equal(f1, phi[sample])
    assert np.array_equal(s1, state[sample])
    for j in range(len(sample)):
        m = (p1[j] if p1[j] >= 0 else n_steps) // 7 + 1
        assert np.all(np.isfinite(path[j, :m])) and np.all(np.isnan(path[j, m:]))


@pytest.mark.parametrize("kw", [dict(s1=0.0, x0=1e-3, y0=0.0), dict(A1=0.0, A3=1e-90), dict(ym=0.4), dict(mass=2.5, gamma=0.3),
                                dict(s_power=2, w=0.0), dict(x0=0.0, y0=0.0, z_product=-1.0), dict(gamma=1e-85)])
@pytest.mark.parametrize("bias", [S.TOY_RATCHET, S.TOY_STEERED])
def test_parameters_outside_the_quotients_range(kw, bias):
    """100 steps against the oracle: only the last bits of the two libraries'
    logarithm and sine differ (1e-16 of a step's noise); 1e-9 of the position
    leaves seven orders for their growth over the run."""
    tp = dataclasses.replace(S.Toy2dParams(), bias=bias, **kw)
    ks, seeds = np.array([0.7, 3.0]), np.array([5, 6], np.uint64)
    _, phi, _, path = B.toy2d_run(tp, ks, seeds, 100, path_every=1)
    for t in range(2):
        _, phr, _, pathr = O.toy2d_run(tp, ks[t], int(seeds[t]), 100, want_path=True)
        scale = max(1.0, np.abs(pathr).max())
        assert np.abs(path[t, :len(pathr)] - pathr).max() <= 1e-9 * scale, t
        assert phi[t] == pytest.approx(phr, rel=1e-6, abs=1e-12)
