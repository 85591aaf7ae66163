"""The integer conversions between FP64 and float-float pairs (csrc/ff_bits.h), compiled
for the host, against the conversions and additions they stand for, bit for bit:
every distance of the two exponents around the line where the sum leaves the integer
arithmetic, both signs, significands at the ends of a binade, and the lines where hi
is too small or too large for it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1010_4782_gb300", "csrc")
SHIM = """
#include <initializer_list>
#include "ff_bits.h"
extern "C" void sums(const float* hi, const float* lo, double* out, long n) {
    for (long k = 0; k < n; ++k) out[k] = stag::ff_sum(hi[k], lo[k]);
}
extern "C" void fixed_sums(const float* s, const float* e, double* out, long n) {  // of 32 pairs each
    for (long k = 0; k < n / 32; ++k) {
        int E = 1;
        for (long j = 32 * k; j < 32 * k + 32; ++j)
            for (float x : {s[j], e[j]})
                if (stag::float_exponent(x) > E) E = stag::float_exponent(x);
        long long v = 0;
        for (long j = 32 * k; j < 32 * k + 32; ++j) v += stag::float_to_fixed(s[j], E) + stag::float_to_fixed(e[j], E);
        out[k] = stag::fixed_to_double(v, E);
    }
}
extern "C" void splits(const double* a, float* hi, float* lo, long n) {
    for (long k = 0; k < n; ++k) {
        const stag::FFPair p = stag::ff_split(a[k]);
        hi[k] = p.hi;
        lo[k] = p.lo;
    }
}
"""


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    d = tmp_path_factory.mktemp("ff_bits")
    src, lib = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(lib)], check=True)
    return ctypes.CDLL(str(lib))


def _call(f, *arrays):
    f(*[ctypes.c_void_p(a.ctypes.data) for a in arrays], ctypes.c_long(arrays[0].size))


MANTISSAS = np.array([0, 1, 2, 0x3FFFFF, 0x400000, 0x400001, 0x600000, 0x7FFFFE, 0x7FFFFF], dtype=np.uint32)


@pytest.mark.parametrize("eh", [1, 23, 39, 40, 41, 64, 127, 128, 250, 251, 254])
def test_sum_of_every_pair_of_edges(shim, eh):
    rng = np.random.default_rng(eh)
    m = np.concatenate([MANTISSAS, rng.integers(0, 1 << 23, 40, dtype=np.uint32)])
    sign = np.array([0, 1], dtype=np.uint32) << np.uint32(31)
    dist = np.array([d for d in (*range(0, 30), 36, 37, 38, 39, 40, 60, 61, 62, 63, 64, 90) if eh - d >= 0])
    hi, lo = [], []
    for d in dist:
        h, l, sh, sl = np.meshgrid(m, m, sign, sign, indexing="ij")
        hi.append((sh | np.uint32(eh << 23) | h).ravel())
        lo.append((sl | np.uint32((eh - int(d)) << 23) | l).ravel())
    zero = np.zeros(m.size, dtype=np.uint32)
    hi += [np.uint32(eh << 23) | m, sign[1] | np.uint32(eh << 23) | m]
    lo += [zero, zero | sign[1]]
    hi, lo = np.concatenate(hi).view(np.float32), np.concatenate(lo).view(np.float32)
    out = np.empty(hi.size)
    _call(shim.sums, hi, lo, out)
    want = hi.astype(np.float64) + lo.astype(np.float64)
    assert np.array_equal(out.view(np.uint64), want.view(np.uint64))


def test_sum_of_specials(shim):
    v = np.array([0.0, -0.0, 1.0, -1.0, 1e-45, -1e-40, 3e38, np.inf, -np.inf, np.nan], dtype=np.float32)
    hi, lo = (np.ascontiguousarray(a.ravel()) for a in np.meshgrid(v, v))
    out = np.empty(hi.size)
    _call(shim.sums, hi, lo, out)
    with np.errstate(invalid="ignore"):
        want = hi.astype(np.float64) + lo.astype(np.float64)
    same = (out.view(np.uint64) == want.view(np.uint64)) | (np.isnan(out) & np.isnan(want))
    assert same.all()


@pytest.mark.parametrize("e", [-1074, -1022, -150, -126, -100, -71, -70, -69, 0, 119, 120, 121, 126, 127, 128, 1023])
def test_split(shim, e):
    rng = np.random.default_rng(e + 2000)
    mant = rng.integers(0, 1 << 52, 4000, dtype=np.uint64)
    mant[1::4] = mant[1::4] >> np.uint64(29) << np.uint64(29) | np.uint64(1 << 28)  # ties
    mant[2::8] &= np.uint64(0xFFFFFFFFFFFFF ^ ((1 << 29) - 1))                       # lo = 0
    mant[3::8] |= np.uint64(0xFFFFFFF000000)                                         # hi to the next binade
    a = np.ldexp(1.0 + mant / 2.0 ** 52, e) * rng.choice([-1.0, 1.0], mant.size)
    a[:4] = [0.0, -0.0, np.inf, -np.inf]
    hi, lo = np.empty(a.size, np.float32), np.empty(a.size, np.float32)
    _call(shim.splits, a, hi, lo)
    with np.errstate(over="ignore", invalid="ignore"):
        h = a.astype(np.float32)
        l = (a - h.astype(np.float64)).astype(np.float32)
    for got, want in ((hi, h), (lo, l)):
        assert ((got.view(np.uint32) == want.view(np.uint32)) | (np.isnan(got) & np.isnan(want))).all()


@pytest.mark.parametrize("spread", [0, 3, 30, 33, 34, 60, 250])
@pytest.mark.parametrize("top", [1, 2, 60, 127, 200, 254])
def test_fixed_point_sum_of_a_warp(shim, top, spread):
    """32 pairs (s, e): exact, then rounded once, when every number is within 2^33 of the
    largest; else each is rounded to 2^-57 of the largest's binade.  Against Fractions; an
    FP64 tree of the same numbers is allowed to be no better in the worst case."""
    from fractions import Fraction
    rng = np.random.default_rng(1000 * top + spread)
    groups = 60
    ex = np.clip(top - rng.integers(0, spread + 1, (groups, 32)), 0, 254).astype(np.uint32)
    ex[:, 0] = top
    s = (ex << np.uint32(23)) | rng.integers(0, 1 << 23, (groups, 32), dtype=np.uint32)
    s[::3] |= rng.integers(0, 2, (len(s[::3]), 32), dtype=np.uint32) << np.uint32(31)  # signs; the others positive
    s[1, 1:] = 0
    s[2] = np.uint32((top << 23) | 0x7FFFFF)   # the largest sum
    s = s.view(np.float32)
    e = (s * rng.uniform(-2.0 ** -23, 2.0 ** -23, s.shape)).astype(np.float32)
    e[2] = s[2]
    out = np.empty(s.size)
    _call(shim.fixed_sums, s.ravel().copy(), e.ravel().copy(), out)
    unit = Fraction(2) ** (top - 127 - 56)
    for k in range(groups):
        numbers = [Fraction(float(v)) for v in (*s[k], *e[k])]
        exact = sum(numbers)
        near = all(v == 0 or abs(v) >= unit * 2 ** 23 for v in numbers)
        slack = Fraction(0) if near else 64 * unit / 2
        got = Fraction(float(out[k]))
        assert abs(got - exact) <= slack + abs(exact) * Fraction(1, 2 ** 53) * Fraction(1001, 1000)
