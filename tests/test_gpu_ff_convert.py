"""Complex FP64 <-> float-float of stag_apply_A: with zero links and mass 1 A is the
identity, so the result is the input after hi = fl32(a), lo = fl32(a - hi) and
hi + lo, bit for bit (the product with the float-float 1 is exact), over signs, rounding
ties, zero low parts, and sizes on both sides of the lines (2^-70, 2^120) where the
conversion changes its form.  NumPy's conversions give the expected bits.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1010_4782_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 2, 10), (8, 8, 6, 12)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("lo_exp,hi_exp", [(-3, 3), (-72, -68), (100, 122)])
def test_identity_through_float_float(dims, lo_exp, hi_exp):
    volume = int(np.prod(dims))
    rng = np.random.default_rng(volume)
    n = volume // 2 * 6
    mant = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    tie = np.arange(n) % 4 == 1  # half of an FP32 unit in the last place exactly
    mant[tie] = mant[tie] >> np.uint64(29) << np.uint64(29) | np.uint64(1 << 28)
    mant[np.arange(n) % 8 == 2] &= np.uint64(0xFFFFFFFFFFFFF ^ ((1 << 29) - 1))  # lo = 0
    mant[np.arange(n) % 8 == 3] |= np.uint64(0xFFFFFFF000000)  # hi rounds up to a power of two
    a = np.ldexp(1.0 + mant / 2.0 ** 52, rng.integers(lo_exp, hi_exp, n)) * rng.choice([-1.0, 1.0], n)
    a[:2] = 0.0
    hi = a.astype(np.float32).astype(np.float64)
    want = hi + (a - hi).astype(np.float32).astype(np.float64)
    opt = binding.stag_default_options()
    opt.arith = binding.STAG_ARITH_FF
    fat = torch.zeros((4, volume, 3, 3), dtype=torch.complex128, device="cuda")
    src = torch.from_numpy(a.view(np.complex128)).cuda()
    out = torch.zeros_like(src)
    with binding.Handle(fat, dims, 1.0, options=opt) as h:
        binding.stag_apply_A(h.h, src, out)
    got = out.cpu().numpy().view(np.float64)
    assert np.array_equal(got, want)
