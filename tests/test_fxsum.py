"""The fixed-point sums of the FP64 kernels (csrc/fv_fxsum.cuh), compiled for
the host, against exact rational arithmetic: every sum that reports itself
exact is the exact sum rounded once to nearest even; sums that would lose
bits, and infinities and NaN, are refused; negating the terms negates it."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2302_09005_gb300 import _build

SRC = """
#include "fv_fxsum.cuh"
template <int N> static void run(const uint64_t* x, long n, uint64_t* out, unsigned char* okv) {
  for (long i = 0; i < n; ++i) {
    uint32_t h[N], l[N], rh, rl;
    for (int k = 0; k < N; ++k) { h[k] = (uint32_t)(x[i * N + k] >> 32); l[k] = (uint32_t)x[i * N + k]; }
    bool ok;
    fv::fx_sum<N, N / 2>(h, l, rh, rl, ok);
    out[i] = ((uint64_t)rh << 32) | rl;
    okv[i] = ok;
  }
}
extern "C" void sum4(const uint64_t* x, long n, uint64_t* o, unsigned char* k) { run<4>(x, n, o, k); }
extern "C" void sum6(const uint64_t* x, long n, uint64_t* o, unsigned char* k) { run<6>(x, n, o, k); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fxsum")
    (d / "t.cpp").write_text(SRC)
    so = str(d / "t.so")
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", _build.CSRC, str(d / "t.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def fx(lib, v):
    n, m = v.shape
    out, ok = np.zeros(n), np.zeros(n, dtype=np.uint8)
    v = np.ascontiguousarray(v)
    getattr(lib, f"sum{m}")(ctypes.c_void_p(v.ctypes.data), ctypes.c_long(n),
                            ctypes.c_void_p(out.ctypes.data), ctypes.c_void_p(ok.ctypes.data))
    return out, ok.astype(bool)


def terms(kind, m, n, rng):
    v = rng.uniform(-1, 1, (n, m))
    if kind == "spread":  # exponents up to 32 apart: some sums are refused
        v = np.ldexp(v, rng.integers(-16, 17, (n, m)))
    elif kind == "cancel":  # plus and minus terms nearly equal
        v[:, m // 2:] = v[:, :m // 2] * (1 + np.ldexp(rng.uniform(-1, 1, (n, m // 2)),
                                                      -rng.integers(0, 54, (n, m // 2))))
    elif kind == "zeros":  # exact zeros of either sign, small integers (ties, carries)
        v = rng.integers(-4, 5, (n, m)).astype(float) * rng.choice([1.0, -1.0], (n, m))
    elif kind == "ties":  # sums half an ulp from a representable number
        v = np.ldexp(1.0 + np.ldexp(rng.integers(0, 8, (n, m)).astype(float), -52),
                     rng.integers(-4, 4, (n, m))) * rng.choice([1.0, -1.0], (n, m))
    elif kind == "ends":  # near the ends of the exponent range
        v = np.ldexp(v, rng.choice([-1070, -1000, -960, -955, 900, 1015, 1020], (n, 1)))
    return v


@pytest.mark.parametrize("m", [4, 6])
@pytest.mark.parametrize("kind", ["plain", "spread", "cancel", "zeros", "ties", "ends"])
def test_exact_or_refused(lib, kind, m):
    rng = np.random.default_rng(m)
    v = terms(kind, m, 4000, rng)
    out, ok = fx(lib, v)
    neg, okn = fx(lib, -v)
    assert np.array_equal(ok, okn) and np.array_equal(out[ok], -neg[ok])
    assert ok.any() or kind == "ends"
    if kind == "plain":  # at most 2^-28 of the draws are small enough to refuse
        assert ok.all()
    for x, r, k in zip(v, out, ok):
        if k:
            s = sum(map(Fraction, x[:m // 2])) - sum(map(Fraction, x[m // 2:]))
            assert r == float(s), (x, r, float(s))


@pytest.mark.parametrize("m", [4, 6])
def test_refuses_what_is_not_exact(lib, m):
    v = np.ones((6, m))
    v[0, 1] = np.inf
    v[1, 0] = np.nan
    v[2, m - 1] = 2.0 ** -29  # would lose bits
    v[3, 0] = 2.0 ** 1020  # beyond what the sum of the others may reach
    v[4, 2] = 2.0 ** -1040
    v[5, 1] = 2.0 ** -28  # the smallest that still fits
    _, ok = fx(lib, v)
    assert ok.tolist() == [False, False, False, False, False, True]
