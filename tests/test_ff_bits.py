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
#include "ff_bits.h"
extern "C" void sums(const float* hi, const float* lo, double* out, long n) {
    for (long k = 0; k < n; ++k) out[k] = stag::ff_sum(hi[k], lo[k]);
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
