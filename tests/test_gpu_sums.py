"""Sums over sites are FP64: a block's or a warp's sum may exceed the FP32 range that the
sites' own numbers stay in.

The source is scaled by a power of two with which one site's d^dag A d is about 2e37 to 1e38
and the sum over the sites of a block (and of a warp where each thread has a site) exceeds
3.4e38.  Scaling by a power of two changes no rounding, so x is the scaled solution of the
unscaled source, bit for bit, after the same number of iterations.
"""
import pytest

torch = pytest.importorskip("torch")
from paper_1010_4782_gb300 import binding as B, inputs  # noqa: E402

pytestmark = pytest.mark.gpu
TOL, MASS = 1e-10, 0.2


def _pair(dims, scale, solve, **kw):
    opt = B.stag_default_options()
    opt.arith = B.STAG_ARITH_FF
    for k, v in kw.items():
        setattr(opt, k, v)
    fat = torch.from_numpy(inputs.gauge_field(dims, 31)).cuda()
    b = torch.from_numpy(inputs.gaussian_even_source(dims, 32)).cuda()
    out = []
    with B.Handle(fat, dims, MASS, options=opt) as h:
        for s in (1.0, scale):
            x = torch.zeros_like(b)
            code, info = solve(h, s * b, x)
            assert code == B.STAG_OK, (s, info)
            out.append((x, info["iters"]))
    assert out[0][1] == out[1][1]
    assert torch.equal(scale * out[0][0], out[1][0])


@pytest.mark.parametrize("inner", [B.STAG_INNER_NONE, B.STAG_INNER_F32, B.STAG_INNER_BF16])
@pytest.mark.parametrize("dims,one_launch", [((10, 6, 4, 12), 0), ((20, 18, 14, 30), 0), ((20, 18, 14, 30), 1),
                                             ((24, 24, 16, 32), 1), ((24, 24, 24, 48), 1)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_solve_of_a_large_source(dims, one_launch, inner):
    """In launches (a lattice of a few blocks, one of many sites a thread, one too large for
    the other way) and in one launch (two and one lanes a site)."""
    def solve(h, b, x):
        B.stag_set_one_launch(h.h, one_launch)
        return B.stag_cg_solve(h.h, b, x, TOL, 20000)

    _pair(dims, 2.0 ** 59, solve, inner=inner)


@pytest.mark.parametrize("form", [B.STAG_PTNET_COLLAPSED, B.STAG_PTNET_LAYERED])
def test_flexible_cg_of_a_large_source(form):
    def solve(h, b, x):
        net = B.stag_ptnet_create(h.h, B.STAG_ARITH_F32, 1)
        try:
            B.stag_ptnet_set_inference_form(net, form)
            return B.stag_fcg_solve(h.h, net, b, x, TOL, 20000)
        finally:
            B.stag_ptnet_destroy(net)

    _pair((10, 6, 4, 12), 2.0 ** 61, solve)


@pytest.mark.parametrize("inner", [B.STAG_INNER_NONE, B.STAG_INNER_F32])
@pytest.mark.parametrize("dims,one_launch", [((10, 6, 4, 12), 0), ((10, 6, 4, 12), 1), ((24, 24, 16, 32), 1)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_sites_beyond_the_range_are_a_breakdown(dims, one_launch, inner):
    """With a site's own |r|^2 beyond the FP32 range the sums are infinite or NaN, and the solve
    ends as a breakdown; the handle's next solve gives the bits of the one before."""
    opt = B.stag_default_options()
    opt.arith, opt.inner = B.STAG_ARITH_FF, inner
    fat = torch.from_numpy(inputs.gauge_field(dims, 31)).cuda()
    b = torch.from_numpy(inputs.gaussian_even_source(dims, 32)).cuda()
    with B.Handle(fat, dims, MASS, options=opt) as h:
        B.stag_set_one_launch(h.h, one_launch)
        xs = []
        for s, want in ((1.0, B.STAG_OK), (2.0 ** 66, B.STAG_ERR_BREAKDOWN), (1.0, B.STAG_OK)):
            x = torch.zeros_like(b)
            assert B.stag_cg_solve(h.h, s * b, x, TOL, 20000, raise_on_error=False)[0] == want
            xs.append(x)
    assert torch.equal(xs[0], xs[2])
