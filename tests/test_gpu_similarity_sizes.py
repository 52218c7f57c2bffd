"""Path similarity at the edges of its kernels: numbers of contacts around the
vector loads and the chunks of the ranking, numbers of distinct times around
the joint histogram's two sizes and the most the device ranks -- the counts
are whole numbers, so every value equals the oracle's."""
import numpy as np
import pytest

import oracle as O
from paper_1405_6104_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1405_6104_gb300 import build
    build.build()
    B.load()


def check(T, pairs):
    got = B.path_similarity(T, pairs)
    clean = np.where(T < 0, -1, T)
    for (a, b), v in zip(pairs, got):
        assert v == O.path_similarity(clean[a], clean[b]), (a, b)


@pytest.mark.parametrize("n_c", [2, 3, 7, 8, 9, 31, 255, 257, 4095, 4096, 4097, 4105])
def test_numbers_of_contacts(n_c):
    rng = np.random.default_rng(n_c)
    T = rng.integers(-1, 12, size=(4, n_c)) * 10
    T[1] = -3                       # nothing formed
    T[2] = np.iinfo(np.int64).max   # the same rank as not formed
    check(T, [(0, 1), (0, 2), (0, 3), (3, 0), (1, 2), (3, 3)])


@pytest.mark.parametrize("ka,kb", [(1, 1), (1, 4096), (64, 64), (65, 64), (128, 32), (13, 315), (230, 231), (231, 231),
                                   (13, 4096), (4096, 14), (1, 4097), (4097, 4097), (2, 5000)])
def test_numbers_of_distinct_times(ka, kb):
    """Both orders of a pair; a few hundred contacts beyond the distinct ones tie."""
    rng = np.random.default_rng(ka * 10007 + kb)
    n_c = max(ka, kb) + 203
    T = np.stack([rng.permutation(np.concatenate([np.arange(k), rng.integers(0, k, n_c - k)])) for k in (ka, kb)])
    assert [len(np.unique(t)) for t in T] == [ka, kb]
    check(T * 977 + (1 << 41), [(0, 1), (1, 0), (0, 0)])


def test_many_paths_in_one_call():
    """More paths than one ranking group holds (256)."""
    rng = np.random.default_rng(3)
    T = rng.integers(-1, 6, size=(300, 40))
    check(T, [(0, 299), (255, 256), (256, 255), (299, 1), (17, 270)])
