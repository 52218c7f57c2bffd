"""The allocation-free reaction coordinate at sizes and parameters where its
tiles can go wrong, against the FP64 oracle."""
import types

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


def _eval(pos, nat, box, p):
    import torch

    dev = torch.device("cuda", 0)
    n = len(pos)
    d_pos = torch.tensor(pos.astype(np.float32).reshape(-1), device=dev)
    d_nat = torch.tensor(np.asarray(nat, np.float64).reshape(-1), device=dev)
    d_z = torch.full((1,), float("nan"), dtype=torch.float64, device=dev)
    d_g = torch.full((3 * n,), float("nan"), dtype=torch.float64, device=dev)
    rc, msg = B.cv_eval_noalloc(d_pos.data_ptr(), d_nat.data_ptr(), n, box, p, d_z.data_ptr(), d_g.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert rc == B.SIM_OK, msg
    return float(d_z.item()), d_g.cpu().numpy().reshape(n, 3)


def _check(pos, nat, box, p):
    """The bounds of the batched kernel: z to 1e-10, the gradient's FP32
    derivatives to 1e-5."""
    z_ref, g_ref = O.cv(types.SimpleNamespace(n_cv=len(pos), native_pos=nat, box=box), p, pos)
    z, g = _eval(pos, nat, box, p)
    assert z == pytest.approx(z_ref, rel=1e-10, abs=1e-10)
    assert np.linalg.norm(g - g_ref) <= 1e-5 * np.linalg.norm(g_ref)
    return z_ref, g_ref


@pytest.mark.parametrize("r0", [1e-8, 1e-7, 1e-6, 1e-3, 0.05])
def test_steep_contacts(r0):
    """Gradient terms up to 1/r0, beyond the tiles' 32-bit halves below r0 =
    1e-5 nm; the sums themselves hold 2^31."""
    rng = np.random.default_rng(9)
    pos = (0.8 * r0 * rng.normal(size=(40, 3))).astype(np.float32).astype(np.float64)
    nat = 3.0 * rng.random((40, 3))
    _, g = _check(pos, nat, 8.0, S.Params(cv_r0=r0, cv_min_sep=2))
    assert np.abs(g).max() > 0.5 / r0


@pytest.mark.parametrize("min_sep", [3, 30, 31, 32, 35, 63, 64])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 36, 37, 64, 65, 97, 540])
def test_tile_edges(n, min_sep):
    """Tile diagonals without a pair left out, partial last tiles, no tile at
    all; 60 atoms per nm^3 (many pairs near)."""
    rng = np.random.default_rng(n)
    pos = (2.0 + (max(n, 30) / 60.0) ** (1.0 / 3.0) * rng.random((n, 3))).astype(np.float32).astype(np.float64)
    z, _ = _check(pos, pos + 0.1 * rng.normal(size=pos.shape), 8.0, S.Params(cv_min_sep=min_sep))
    assert (z > 0.0) == (n > min_sep + 1)


def test_no_atom():
    z, g = _eval(np.zeros((0, 3)), np.zeros((0, 3)), 8.0, S.Params())
    assert z == 0.0 and g.shape == (0, 3)


@pytest.mark.parametrize("shift", [0.0, 1000.0])
def test_native_pairs_around_the_cut_off(shift):
    """Native distances within 3e-3 nm of the cut-off (the FP32 test of the
    native structure passes pairs up to 4e-3 nm beyond), the structure far
    from the origin; a narrow switch, so that C~ is visible next to it."""
    rng = np.random.default_rng(11)
    p = S.Params(cv_min_sep=2, cv_r_switch=1.19)
    nat = np.zeros((70, 3))
    nat[:35] = 0.05 * rng.normal(size=(35, 3))
    u = rng.normal(size=(35, 3))
    nat[35:] = nat[:35] + (p.cv_r_cut + 3e-3 * rng.uniform(-1, 1, (35, 1))) * u / np.linalg.norm(u, axis=1)[:, None]
    pos = (3.0 + 0.4 * rng.normal(size=(70, 3))).astype(np.float32).astype(np.float64)
    _check(pos, nat + shift, 8.0, p)
