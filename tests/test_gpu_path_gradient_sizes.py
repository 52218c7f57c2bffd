"""Sizes at which the kernels of the path gradient can go wrong: the scan of
the coefficients at the edges of its warps and of its chunks of frames, and
the tile kernels in their two forms (a block or a warp per tile), which must
agree bit for bit; contacts too steep for the tiles' 32-bit accumulators."""
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


def coefficients(z, Q, c):
    """The definition, frame by frame (FP64)."""
    n = len(z)
    coef, route = np.zeros((n, 2)), np.zeros(n)
    m, arg, phi = z[0], 0, 0.0
    for f in range(1, n):
        a = z[f] - m if z[f] > m else 0.0
        phi += c * a * a * Q[f]
        if a > 0.0:
            route[arg] += 2.0 * a * Q[f]
        coef[f] = 2.0 * c * a * Q[f], 2.0 * c * a * a
        if z[f] < m:
            m, arg = z[f], f
    coef[:, 0] -= c * route
    return coef, phi


@pytest.mark.parametrize("shape", ["falling", "rising", "walk", "flat", "late"])
@pytest.mark.parametrize("n", [1, 2, 32, 33, 34, 1024, 1025, 1026, 2500])
def test_coefficients_at_the_edges_of_the_scan(n, shape):
    """Sums of up to n terms of one sign in two orders differ by at most
    about n 2^-53 relative (n = 2500: 3e-13); 1e-12 bounds them."""
    rng = np.random.default_rng(n)
    z = {"falling": -np.arange(n, dtype=float), "rising": np.arange(n, dtype=float), "flat": np.full(n, 3.0),
         "walk": rng.normal(size=n).cumsum(), "late": np.where(np.arange(n) == n - 1, -1.0, rng.random(n))}[shape]
    Q = rng.random(n) + 0.5
    s, p = S.tiny_chain(0)
    with B.TrialBatch(s, p, [1]) as b:
        coef, phi = B.phi_adjoint_coefficients(b.h, z, Q)
    ref, phi_ref = coefficients(z, Q, p.dt * (0.5 * p.k_ratchet) ** 2)
    np.testing.assert_allclose(coef, ref, rtol=1e-12, atol=0.0)
    assert phi == pytest.approx(phi_ref, rel=1e-12, abs=0.0)


@pytest.mark.parametrize("n_solute", [12, 33, 64, 97])
def test_tiles_by_a_block_match_tiles_by_a_warp(n_solute):
    """The same frames in a short call (few tiles: a block each) and among
    many (a warp each), with given coefficients: equal bits of z and of the
    gradient, for tiles near, partly filled and far apart."""
    s, p = S.small_solvated(n_solute=n_solute, n_water=430 + n_solute)
    rng = np.random.default_rng(n_solute)
    base = s.native_pos + 0.3 * rng.normal(size=(1, 3))
    frames = np.stack([base * f for f in (0.4, 1.0, 2.5)]) + 0.01 * rng.normal(size=(3, n_solute, 3))
    coef = rng.normal(size=(3, 2))
    tiles = ((n_solute + 31) // 32) * ((n_solute + 31) // 32 + 1) // 2
    reps = 128 * 160 // (3 * tiles) + 2  # beyond 128 tiles per multiprocessor
    with B.TrialBatch(s, p, [1]) as b:
        _, z, g = B.phi_frames_adjoint(b.h, 0, frames, coef)
        _, zz, gg = B.phi_frames_adjoint(b.h, 0, np.concatenate([frames] * reps), np.concatenate([coef] * reps))
    assert np.abs(g).max() > 0.0
    assert (zz.reshape(reps, 3) == z).all() and (gg.reshape(reps, *g.shape) == g).all()


@pytest.mark.parametrize("n_solute", [12, 33])
def test_near_pairs_kept_match_near_pairs_listed_again(n_solute):
    """Beyond 500 000 tiles the second pass lists the near pairs itself: equal
    bits with a short call, whose first pass keeps them."""
    s, p = S.small_solvated(n_solute=n_solute, n_water=430 + n_solute)
    rng = np.random.default_rng(n_solute)
    frames = s.native_pos * np.array([0.4, 1.0, 2.5])[:, None, None] + 0.01 * rng.normal(size=(3, n_solute, 3))
    coef = rng.normal(size=(3, 2))
    reps = 500_000 // (3 * (1 if n_solute <= 32 else 3)) + 2
    with B.TrialBatch(s, p, [1]) as b:
        _, z, g = B.phi_frames_adjoint(b.h, 0, frames, coef)
        _, zz, gg = B.phi_frames_adjoint(b.h, 0, np.concatenate([frames] * reps), np.concatenate([coef] * reps))
    assert np.abs(g).max() > 0.0
    assert (zz.reshape(reps, 3) == z).all() and (gg.reshape(reps, *g.shape) == g).all()


@pytest.mark.parametrize("r0", [1e-3, 0.05])
def test_steep_contacts(r0):
    """Contacts so steep that a pair's gradient and Hessian terms pass the
    range of the tiles' 32-bit accumulators, against the FP64 oracle; the
    bounds are those of ordinary contacts (FP32 derivatives of C~).  r0 = 1e-3
    nm: gradients of 1e3, checked through Phi = sum a^2 |grad z|^2 only, as the
    Hessian products (1e10) leave the range +-2^31 of the 64-bit sums; r0 =
    0.05 nm: Hessian products of 1e5."""
    s, p = S.tiny_chain(0)
    p.cv_r0 = r0
    rng = np.random.default_rng(4)
    frames = s.native_pos * np.array([1.0, 0.02, 0.01, 0.004])[:, None, None] * (r0 / 0.01)
    frames = (frames + 0.3 * r0 * rng.normal(size=frames.shape)).astype(np.float32).astype(np.float64)
    with B.TrialBatch(s, p, [1]) as b:
        phi, z, G = B.phi_frames_adjoint(b.h, 0, frames)
    phi_ref, G_ref = O.phi_frames_grad(s, p, frames)
    _, z_ref, _, _ = O.phi_frames(s, p, frames)
    assert phi_ref > 0
    assert phi == pytest.approx(phi_ref, rel=1e-5)
    assert np.allclose(z, z_ref, rtol=1e-11, atol=1e-11)
    if r0 > 1e-3:
        assert np.linalg.norm(G - G_ref) < 1e-4 * np.linalg.norm(G_ref)
