"""The quotients and roots that the reaction coordinate's kernels form from an
approximate reciprocal (vp_cvpair.cuh), against CUDA's operators: all
significands, random operands, operands whose exact result lies next to the
midpoint of two numbers, and the ends of the stated ranges.  The functions are
compiled from the kernels' own source."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1405_6104_gb300 import build as _build

pytestmark = pytest.mark.gpu

F32 = r"""
#include "vp_cvpair.cuh"
using namespace vp;
__global__ void k32(int op, const float *a, const float *b, float *got, float *ref, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const float2 x = make_float2(a[i], a[n - 1 - i]), y = make_float2(b[i], b[n - 1 - i]);
  const float2 r = op == 0 ? f2_rcp(y) : op == 1 ? f2_div(x, y, f2_rcp(y)) : f2_sqrt(y);
  got[i] = r.x;
  ref[i] = op == 0 ? 1.0f / y.x : op == 1 ? x.x / y.x : sqrtf(y.x);
}
template <bool SECOND>
__global__ void kc(CvConst k, const float *r2, float *out, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const CvPair2 p = cv_contact2<SECOND>(ff2{make_float2(r2[i], r2[n - 1 - i]), make_float2(0.f, 0.f)}, k);
  out[3 * i] = p.Ct.hi.x;
  out[3 * i + 1] = p.dCt.x;
  out[3 * i + 2] = SECOND ? p.d2Ct.x : 0.f;
}
extern "C" __attribute__((visibility("default"))) int run32(int op, const float *a, const float *b, float *got, float *ref, int n) {
  k32<<<(n + 255) / 256, 256>>>(op, a, b, got, ref, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" __attribute__((visibility("default"))) int contact32(int second, double r0, double rs, double rc, const float *r2, float *out, int n) {
  auto split = [](double v) { const float h = (float)v; return ff{h, (float)(v - (double)h)}; };
  const CvConst k{split(1.0 / (r0 * r0)), split(rs), split(1.0 / (rc - rs)), (float)(rs * rs), (float)(rc * rc * (1.0 + 1e-4)),
                  rc * rc > 1000.0 * r0 * r0};
  if (second) kc<true><<<(n + 255) / 256, 256>>>(k, r2, out, n);
  else kc<false><<<(n + 255) / 256, 256>>>(k, r2, out, n);
  return (int)cudaDeviceSynchronize();
}
"""


def compiled(d, name, src, flags=()):
    (d / f"{name}.cu").write_text(src)
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, *flags, "-I", _build.SRC, "-shared",
                    str(d / f"{name}.cu"), "-o", str(d / f"{name}.so")], check=True, cwd=_build.SRC)
    return ctypes.CDLL(os.fspath(d / f"{name}.so"))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return compiled(tmp_path_factory.mktemp("rounding"), "f32", F32)


def run(fn, op, a, b, dtype):
    import torch

    a, b = (torch.tensor(np.ascontiguousarray(v, dtype), device="cuda") for v in (a, b))
    got, ref = torch.empty_like(b), torch.empty_like(b)
    rc = fn(op, *(ctypes.c_void_p(t.data_ptr()) for t in (a, b, got, ref)), b.numel())
    assert rc == 0
    return got.cpu().numpy(), ref.cpu().numpy()


def same(got, ref):
    return np.array_equal(got.view(np.int32 if got.dtype == np.float32 else np.int64),
                          ref.view(np.int32 if ref.dtype == np.float32 else np.int64))


@pytest.mark.parametrize("exponent", [-126, -125, 0, 1, 125])
def test_reciprocals_of_every_significand(lib, exponent):
    b = np.ldexp(np.arange(1 << 23, 1 << 24).astype(np.float32), exponent - 23).astype(np.float32)
    assert same(*run(lib.run32, 0, b, b, np.float32))


@pytest.mark.parametrize("exponent", [-100, -99, 0, 1, 126])
def test_fp32_roots_of_every_significand(lib, exponent):
    x = np.ldexp(np.arange(1 << 23, 1 << 24).astype(np.float32), exponent - 23).astype(np.float32)
    assert same(*run(lib.run32, 2, x, x, np.float32))


def hard_quotients(divisors, bits, residues):
    """Pairs (A, B, k, c) of integers of `bits` bits with A 2^k = B (2M + 1) + c:
    A/B lies c/(2B) of a unit in the last place off a midpoint."""
    out = []
    for B in divisors:
        for k in (bits, bits + 1):
            inv = pow(2, -k, B)
            for c in residues:
                A = c * inv % B
                while A < 1 << bits:
                    if A >= 1 << (bits - 1) and (A >= B) == (k == bits) and ((A << k) - c) // B & 1:
                        out.append((A, B, k, c))
                    A += B
    return out


def test_fp32_quotients(lib):
    rng = np.random.default_rng(1)
    n = 1 << 22
    a, b = (rng.choice([-1.0, 1.0], n) * np.ldexp(1.0 + rng.random(n), rng.integers(-40, 40, n)) for _ in range(2))
    assert same(*run(lib.run32, 1, a, np.abs(b), np.float32))
    hard = hard_quotients([int(B) | 1 for B in rng.integers(1 << 23, 1 << 24, 20000)] +
                           [(1 << 24) - q for q in range(1, 400, 2)], 24, (-5, -3, -2, -1, 1, 2, 3, 5))
    a, b = (np.array(v, np.float32) for v in ([h[0] for h in hard], [h[1] for h in hard]))
    assert len(hard) > 10000 and same(*run(lib.run32, 1, a, b, np.float32))


@pytest.mark.parametrize("second", [0, 1])
@pytest.mark.parametrize("r0", [0.75, 0.05, 0.025, 0.02, 4e-3, 1e-3, 1e-4])
def test_contacts_far_beyond_their_radius(lib, r0, second):
    """C, dC/dr and d2C/dr2 at distances up to 1.1 nm, 11 000 r0: D^2 and D^3
    of the derivatives' denominators leave the FP32 range.  A term of C' or C''
    takes some 20 roundings of 2^-24 and the distance's own, amplified at most
    12 times in t^12: 40 units of 2^-24 of the terms' absolute sum."""
    import torch

    rng = np.random.default_rng(7)
    r2 = np.exp(rng.uniform(np.log((0.5 * r0) ** 2), np.log(1.1 ** 2), 20000)).astype(np.float32)
    d = torch.tensor(r2, device="cuda")
    out = torch.empty((len(r2), 3), dtype=torch.float32, device="cuda")
    assert lib.contact32(second, ctypes.c_double(r0), ctypes.c_double(1.2), ctypes.c_double(1.5),
                            ctypes.c_void_p(d.data_ptr()), ctypes.c_void_p(out.data_ptr()), len(r2)) == 0
    got = out.cpu().numpy().astype(np.float64)
    r = np.sqrt(r2.astype(np.float64))
    t = (r / r0) ** 2
    N, N1, N2 = 1 + t + t ** 2, 1 + 2 * t, 2.0
    D, D1, D2 = N + t ** 3 + t ** 4, N1 + 3 * t ** 2 + 4 * t ** 3, 2 + 6 * t + 12 * t ** 2
    ds, dds = 2 * r / r0 ** 2, 2 / r0 ** 2
    b, a = N1 / D, N / D * (D1 / D)
    eps = 40 * 2.0 ** -24
    assert np.all(np.abs(got[:, 0] - N / D) <= 1e-6 * N / D)
    assert np.all(np.abs(got[:, 1] - (b - a) * ds) <= eps * (b + a) * ds)
    if second:
        p, e, q = N2 / D, N / D * (D2 / D), 2 * D1 / D
        exact = (p - e - q * (b - a)) * ds ** 2 + (b - a) * dds
        assert np.all(np.abs(got[:, 2] - exact) <= eps * ((p + e + q * (b + a)) * ds ** 2 + (b + a) * dds))
