"""Fig. 1 in one launch (small lattices): the first iterates against the oracle's CG,
on sizes at the edges of the kernel's forms (8, 4, 2 and 1 lanes per site, V/2 not a
multiple of a warp's sites, more iterations than one block of check_interval) and
just above the largest size it takes.

Bounds: four iterations from x = 0 amplify a relative rounding u of A by at most a few
tens (the iterates are polynomials of A of degree 3 with coefficients of order one on
these spectra): 64 u with u = 2^-48 for float-float (FP64 is below it) and 2^-24 for FP32.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1010_4782_gb300 import binding, inputs  # noqa: E402

pytestmark = pytest.mark.gpu
ITERS = 4
BOUND = {"f64": 64 * 2.0 ** -48, "ff": 64 * 2.0 ** -48, "f32": 64 * 2.0 ** -24}


def _iterate(form, fat, lng, dims, mass, b, **kw):
    opt = binding.stag_default_options()
    opt.arith = binding.STAG_ARITH_F64 if form == "f64" else binding.STAG_ARITH_FF
    opt.inner = binding.STAG_INNER_F32 if form == "f32" else binding.STAG_INNER_NONE
    for k, v in kw.items():
        setattr(opt, k, v)
    bd = torch.from_numpy(b).cuda()
    x = torch.zeros_like(bd)
    naik = None if lng is None else torch.from_numpy(lng).cuda()
    with binding.Handle(torch.from_numpy(fat).cuda(), dims, mass, naik_long=naik, options=opt) as h:
        code, info = binding.stag_cg_solve(h.h, bd, x, 1e-14, ITERS)
        launches = binding.stag_launch_count(h.h)
    assert code == binding.STAG_ERR_NOT_CONVERGED and info["iters"] == ITERS
    return x.cpu().numpy().reshape(-1), launches


# V/2: 24, 60, 1440, 4860 | 5040 (FP32: 8 | 4 lanes), 9720 | 9744 (FP64 class: 8 | 4),
# 37800 (2), 75600 (FP32 2, FP64 class 1), 147456 (FP32 1; FP64 class: launches)
SIZES = [(2, 2, 2, 6), (6, 2, 2, 10), (10, 6, 4, 12), (18, 6, 6, 30), (10, 12, 6, 28), (18, 12, 6, 30),
         (14, 12, 4, 58), (14, 18, 10, 30), (20, 18, 14, 30), (24, 24, 16, 32)]


@pytest.mark.parametrize("form", ["f64", "ff", "f32"])
@pytest.mark.parametrize("naik", [False, True])
@pytest.mark.parametrize("dims", SIZES, ids=lambda d: "x".join(map(str, d)))
def test_first_iterates_match_the_oracle(dims, naik, form):
    if naik:
        fat, lng = inputs.asqtad_form_fields(dims, seeds=(41, 42, 43))
    else:
        fat, lng = inputs.gauge_field(dims, 41), None
    b = inputs.gaussian_even_source(dims, 44)
    x, _ = _iterate(form, fat, lng, dims, 0.1, b)
    ref = oracle.cg_fig1(oracle.Operator(fat, lng, 0.1, dims).apply_A, b, np.zeros_like(b), 1e-14, ITERS)[0]
    assert np.linalg.norm(x - ref) <= BOUND[form] * np.linalg.norm(ref)


@pytest.mark.parametrize("form", ["f64", "ff"])
def test_one_launch_per_run_and_any_block_length(form):
    """The iterations are one launch, and check_interval does not change FP64's bits."""
    dims = (8, 6, 4, 10)
    fat = inputs.gauge_field(dims, 45)
    b = inputs.gaussian_even_source(dims, 46)
    x, few = _iterate(form, fat, None, dims, 0.1, b)
    y, same = _iterate(form, fat, None, dims, 0.1, b, check_interval=3)
    assert few == same  # four iterations, one launch either way
    if form == "f64":
        assert np.array_equal(x, y)
    else:
        assert np.linalg.norm(x - y) <= 4 * 2.0 ** -48 * np.linalg.norm(x)
