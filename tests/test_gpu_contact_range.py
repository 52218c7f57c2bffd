"""Contact parameters and frames at the ends of what the path gradient takes:
pairs at distances far beyond a small contact radius, or next to none, against
the FP64 oracle."""
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


def _check(s, p, frames):
    """The bounds of ordinary contacts (FP32 derivatives of C~)."""
    phi_ref, G_ref = O.phi_frames_grad(s, p, frames)
    _, z_ref, a_ref, _ = O.phi_frames(s, p, frames)
    assert a_ref.max() > 0.1 and phi_ref > 0
    with B.TrialBatch(s, p, [1]) as b:
        phi, z, G = B.phi_frames_adjoint(b.h, 0, frames)
    assert phi == pytest.approx(phi_ref, rel=1e-5)
    assert np.allclose(z, z_ref, rtol=1e-11, atol=1e-11)
    assert np.linalg.norm(G - G_ref) < 1e-4 * np.linalg.norm(G_ref)


@pytest.mark.parametrize("r0", [0.02, 0.025, 4e-3])
def test_pairs_far_beyond_the_contact_radius(r0):
    """Two groups of six beads 1 nm apart (near pairs at 35 to 300 contact
    radii); in the second frame two beads of one group come within a radius of
    each other, so that z rises and the Hessian product is taken."""
    s, p = S.tiny_chain(0)
    p.cv_r0 = r0
    rng = np.random.default_rng(5)
    x = 0.12 * rng.normal(size=(s.n_cv, 3)) * np.array([0.3, 1.0, 1.0]) + 1.0
    x[6:, 0] += 1.02
    frames = np.stack([x, x, x])
    frames[1, 4] = frames[1, 0] + 1.1 * r0 * np.array([0.6, 0.64, 0.48])
    frames[2, 5] = frames[2, 1] + 1.3 * r0 * np.array([0.48, 0.6, 0.64])
    frames = frames.astype(np.float32).astype(np.float64)
    d = np.linalg.norm(frames[1, :6, None] - frames[1, None, 6:], axis=2)
    assert ((d > 0.9) & (d < 1.2) & (d > 40 * r0)).sum() > 5
    _check(s, p, frames)


def test_atoms_that_all_but_coincide():
    """1e-20 nm apart (r^2 below the normal FP32 range): the oracle's gradient;
    exactly at one place: the same, C' and C'' vanish there."""
    s, p = S.tiny_chain(0)
    rng = np.random.default_rng(6)
    frames = np.stack([s.native_pos * f for f in (1.0, 0.7, 0.8)]) + 0.02 * rng.normal(size=(3, s.n_cv, 3))
    frames = frames.astype(np.float32).astype(np.float64)
    frames[1, [0, 6]] = 0.0
    frames[1, 6, 1] = 1e-20
    _check(s, p, frames)
    with B.TrialBatch(s, p, [1]) as b:
        _, z, G = B.phi_frames_adjoint(b.h, 0, frames)
        frames[1, 6, 1] = 0.0
        _, z0, G0 = B.phi_frames_adjoint(b.h, 0, frames)
    assert np.array_equal(z, z0) and np.array_equal(G, G0)
