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
