"""Contact parameters and frames at the ends of what the path gradient takes:
pairs at distances far beyond a small contact radius, or next to none, against
the FP64 oracle."""
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


def _frames_near_the_cut_off(s, p, rng, n):
    """Two compact groups of atoms (points 1/64 nm apart, which the FP32 spacing of
    1/128 at 1e5 nm keeps distinct) whose mutual distances lie around the contact cut-off,
    in random orientations."""
    half = s.n_cv // 2
    out = []
    for _ in range(n):
        q = np.concatenate([rng.choice(125, k, replace=False) for k in (half, s.n_cv - half)])
        x = (np.stack([q // 25, q // 5 % 5, q % 5], axis=1) - 2.0 + 0.25 * rng.random((s.n_cv, 3))) / 64.0
        u = rng.normal(size=3)
        x[half:] += (p.cv_r_cut - 0.012) * u / np.linalg.norm(u)
        out.append(x + s.box / 2)
    return np.stack(out)


@pytest.mark.parametrize("where", ["mixed", "all"])
@pytest.mark.parametrize("boxes", [1, 2 ** 7, 2 ** 15])
def test_atoms_many_boxes_away(boxes, where):
    """Half of the atoms, or all, 2^15 boxes from the origin: the FP32 tests that
    sort out far pairs and far tiles round coordinates of 1e5 nm by 4e-3 nm."""
    import torch

    s, p = S.small_solvated(n_solute=64, n_water=494)
    frames = _frames_near_the_cut_off(s, p, np.random.default_rng(12), 24)
    frames[:, s.n_cv // 2 if where == "mixed" else 0:] += boxes * float(np.float32(s.box))
    frames = frames.astype(np.float32).astype(np.float64)
    coef = np.random.default_rng(13).normal(size=(len(frames), 2))
    _, z_ref, _, _ = O.phi_frames(s, p, frames)
    with B.TrialBatch(s, p, [1]) as b:
        _, z, g = B.phi_frames_adjoint(b.h, 0, frames, coef)
        _, z1, g1 = B.phi_frames_adjoint(b.h, 0, np.tile(frames, (300, 1, 1)), np.tile(coef, (300, 1)))
    assert np.allclose(z, z_ref, rtol=1e-11, atol=1e-11)
    assert np.array_equal(z1[:len(z)], z) and np.array_equal(g1[:len(z)], g)
    for f in range(0, len(frames), 6):
        z0, g0 = O.cv(types.SimpleNamespace(n_cv=s.n_cv, native_pos=s.native_pos, box=s.box), p, frames[f])
        dev = torch.device("cuda", 0)
        d_pos = torch.tensor(frames[f].astype(np.float32).reshape(-1), device=dev)
        d_nat = torch.tensor(np.asarray(s.native_pos, np.float64).reshape(-1), device=dev)
        d_z, d_g = (torch.zeros(k, dtype=torch.float64, device=dev) for k in (1, 3 * s.n_cv))
        rc, msg = B.cv_eval_noalloc(d_pos.data_ptr(), d_nat.data_ptr(), s.n_cv, s.box, p, d_z.data_ptr(), d_g.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)
        assert rc == B.SIM_OK, msg
        assert float(d_z.item()) == pytest.approx(z0, rel=1e-10, abs=1e-10)
        assert np.linalg.norm(d_g.cpu().numpy().reshape(-1, 3) - g0) <= 1e-5 * np.linalg.norm(g0)
