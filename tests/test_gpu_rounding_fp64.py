"""The FP64 quotients and roots of the toy model's kernels (vp_toy2d.cu),
against CUDA's operators: random operands, operands whose exact result lies
next to the midpoint of two numbers, and halving.  The functions are compiled
from the kernels' own source."""
import numpy as np
import pytest
from test_gpu_rounding import compiled, hard_quotients, run, same

from paper_1405_6104_gb300 import build as _build

pytestmark = pytest.mark.gpu

F64 = r"""
#include "vp_toy2d.cu"
using namespace vp;
__global__ void k64(int op, const double *a, const double *b, double *got, double *ref, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const double x = a[i], y = b[i];
  got[i] = op == 0 ? quotient(x, y, reciprocal(y)) : op == 1 ? root(y, inv_sqrt(y)) : op == 2 ? half_of(y) : op == 3 ? reciprocal(y) : inv_sqrt(y);
  ref[i] = op == 0 ? x / y : op == 1 ? sqrt(y) : op == 2 ? 0.5 * y : op == 3 ? 1.0 / y : 1.0 / sqrt(y);
}
extern "C" __attribute__((visibility("default"))) int run64(int op, const double *a, const double *b, double *got, double *ref, int n) {
  k64<<<(n + 255) / 256, 256>>>(op, a, b, got, ref, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return compiled(tmp_path_factory.mktemp("rounding"), "f64", F64, _build.EXTRA["vp_toy2d.cu"])


@pytest.mark.parametrize("exponent", [-300, -1, 0, 299])
def test_every_leading_word(lib, exponent):
    """The approximations see the leading word of a number: over all of them
    the reciprocal and the inverse root are within one ulp and two (the
    reference's own two roundings included), quotients and roots the operators'."""
    rng = np.random.default_rng(abs(exponent))
    high = np.repeat(np.arange(1 << 20, dtype=np.int64) << 32, 3)
    low = np.tile(np.array([0, 0xffffffff, 0], np.int64), 1 << 20)
    low[2::3] = rng.integers(0, 1 << 32, 1 << 20)
    b = ((np.int64(1023 + exponent) << 52) | high | low).view(np.float64)
    a = 1.0 + rng.random(len(b))
    for op, ulps in ((0, 0), (1, 0), (3, 1), (4, 2)):
        got, ref = run(lib.run64, op, a, b, np.float64)
        assert np.abs(got.view(np.int64) - ref.view(np.int64)).max() <= ulps, op


def test_fp64_quotients(lib):
    """Equal to the operator on random operands; next to a midpoint within
    1/2 + 2^-51 of a unit in the last place (the reciprocal is an ulp off at
    most, the quotient before the last step two)."""
    rng = np.random.default_rng(2)
    n = 1 << 22
    a, b = (rng.choice([-1.0, 1.0], n) * np.ldexp(1.0 + rng.random(n), rng.integers(-100, 100, n)) for _ in range(2))
    assert same(*run(lib.run64, 0, a, np.abs(b), np.float64))
    hard = hard_quotients([int(B) | 1 for B in rng.integers(1 << 52, 1 << 53, 3000)] +
                           [(1 << 53) - q for q in list(range(1, 2000, 2)) + [0x44b9]], 53, (-9, -4, -2, -1, 1, 2, 4, 9))
    hard.append((0x132f55cf051791, 0x1fffffffffbb47, None, None))
    got, _ = run(lib.run64, 0, [h[0] for h in hard], [h[1] for h in hard], np.float64)
    assert len(hard) > 10000
    wrong = 0
    for (A, B, k, _), g in zip(hard, got):
        k = 52 if A >= B else 53  # the quotient's last place is 2^-k
        Q = int(g * 2.0 ** k)
        assert Q == g * 2.0 ** k
        off = abs((A << k) - B * Q)  # of a unit in the last place: off / B
        assert 2 * off * 2 ** 50 <= B * (2 ** 50 + 1), (A, B, Q)
        wrong += 2 * off > B
    print(f"quotients next to a midpoint rounded to its other side: {wrong} of {len(hard)}")


def test_fp64_roots_and_halves(lib):
    rng = np.random.default_rng(3)
    n = 1 << 22
    x = np.ldexp(1.0 + rng.random(n), rng.integers(-200, 200, n))
    assert same(*run(lib.run64, 1, x, x, np.float64))
    assert same(*run(lib.run64, 2, x, x, np.float64))
    # s^2 + c = X 2^55 with s odd: sqrt(X 2^55)/2 lies c/(4 s) of a unit off the midpoint s/2
    hard = []
    for d in range(1, 40000, 8):  # s^2 = d mod 2^55
        for sign in (1, -1):
            t = d if sign > 0 else (1 << 55) - (d + 6)  # 1 modulo 8 either way
            s = 1
            for bit in range(3, 56):  # lifts a root modulo 2^bit to one modulo 2^(bit + 1)
                if (s * s - t) >> bit & 1:
                    s += 1 << (bit - 1)
            for q in (s, (1 << 55) - s, (s + (1 << 54)) % (1 << 55), ((1 << 54) - s) % (1 << 55)):
                if not 1 << 53 <= q < 1 << 54:
                    continue
                c = -d if sign > 0 else d + 6
                if (q * q + c) % (1 << 55) == 0 and (q * q + c) >> 55 < 1 << 53:
                    hard.append(((q * q + c) >> 55, q, c))
    assert len(hard) > 1000
    # X 2^55 = (X 2) 2^54: the root of 2 X is 2^-27 of the integer root
    got, _ = run(lib.run64, 1, [0.0] * len(hard), [2.0 * h[0] for h in hard], np.float64)
    wrong = 0
    for (X, s, c), g in zip(hard, got):
        Q = int(g * 2.0 ** 26)  # of sqrt(X 2^55)/2
        assert Q == g * 2.0 ** 26 and abs(2 * Q - s) == 1, (X, s, c)
        if (2 * Q > s) != (c > 0):
            wrong += 1
            assert abs(c) << 51 <= 4 * s, (X, s, c)
    print(f"roots next to a midpoint rounded to its other side: {wrong} of {len(hard)}")
