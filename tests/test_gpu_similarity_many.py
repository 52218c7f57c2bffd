"""Path similarity from all ordered contact pairs with as many paths as their
ranks find room for in the times' place (512), and more."""
import numpy as np
import pytest
from test_gpu_similarity_sizes import _lib, check  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_paths", [2, 300, 512, 513])
def test_all_ordered_pairs_of_many_paths(n_paths):
    """Paths ranked on the device (some hundred distinct times) and on the host
    (more than 4096), in every place."""
    rng = np.random.default_rng(n_paths)
    n_c = 4300
    T = rng.integers(-1, 400, size=(n_paths, n_c)) * 10
    T[1::7] = rng.permuted(np.tile(np.arange(n_c), (len(T[1::7]), 1)), axis=1) * 3
    last = n_paths - 1
    check(T, [(0, 1), (1, 0), (last, 0), (1, last), (last // 2, last), (0, 0)])
