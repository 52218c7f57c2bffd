"""The path gradient written over the frames it is taken at."""
import numpy as np
import pytest

from paper_1405_6104_gb300 import binding as B
from paper_1405_6104_gb300 import systems as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pinned", [False, True])
def test_gradient_over_its_frames(pinned):
    """With work still queued on the caller's stream, so that an asynchronous
    copy of the frames (from page-locked memory) waits while the call goes on:
    the same bits as into an array of its own."""
    import torch

    from paper_1405_6104_gb300 import build
    build.build()
    s, p = S.small_solvated(n_solute=97, n_water=527)
    rng = np.random.default_rng(8)
    frames = s.native_pos * np.array([0.4, 1.0, 2.5, 0.8])[:, None, None] + 0.01 * rng.normal(size=(4, 97, 3))
    frames = np.tile(frames, (50, 1, 1))
    coef = rng.normal(size=(len(frames), 2))
    stream = torch.cuda.Stream()
    x = torch.empty(frames.shape, dtype=torch.float64, pin_memory=pinned).numpy()
    with B.TrialBatch(s, p, [1], cuda_stream=stream.cuda_stream) as b:
        _, z, g = B.phi_frames_adjoint(b.h, 0, frames, coef)
        assert np.abs(g).max() > 0.0
        x[:] = frames
        with torch.cuda.stream(stream):
            torch.cuda._sleep(40_000_000)  # about 20 ms
        _, zz, gg = B.phi_frames_adjoint(b.h, 0, x, coef, out=x)
    assert gg is x and np.array_equal(zz, z) and np.array_equal(gg, g)
