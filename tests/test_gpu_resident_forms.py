"""The one-launch CG in every storage form, over more iterations than one launch holds, and
from two threads at once.

Iterates of every form against the same iterations in launches, at sizes that take eight,
four (512 and 1024 threads a block), two and one lanes a site.  Both ways round the
same stored numbers; their FP32 (float-float) sums differ in order, by about 2^-22 (2^-46) of
a number.  In FP32 and float-float storage three iterations amplify that by at most a few
tens: 64 units of 2^-24 (2^-48).  A number stored with spacing s may then fall on the other
side of a rounding line with probability 2^-22 / s, which moves it by s: sqrt(2^-22 s) rms,
times the same 64.  Against the oracle: 64 units of the storage's rounding more.
"""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1010_4782_gb300 import binding as B, inputs  # noqa: E402

pytestmark = pytest.mark.gpu
FF, F64 = B.STAG_ARITH_FF, B.STAG_ARITH_F64
ROWS = dict(long_recon=12, long_scale=inputs.NAIK_COEFF)
STORED = {8: 64 * (2.0 ** -22 * 2.0 ** -8) ** 0.5, 11: 64 * (2.0 ** -22 * 2.0 ** -11) ** 0.5,
          24: 64 * 2.0 ** -24, 48: 64 * 2.0 ** -48}
# name: (options, Naik, significand bits of the vectors, of the links)
FORMS = {
    "ff_rows": (dict(arith=FF, **ROWS), True, 48, 48),
    "f32_rows_fat": (dict(arith=FF, inner=B.STAG_INNER_F32, link_recon=12), False, 24, 24),
    "f32_rows_naik": (dict(arith=FF, inner=B.STAG_INNER_F32, **ROWS), True, 24, 24),
    "f16": (dict(arith=FF, inner=B.STAG_INNER_F16), False, 11, 11),
    "f16_naik": (dict(arith=FF, inner=B.STAG_INNER_F16), True, 11, 11),
    "b16": (dict(arith=FF, inner=B.STAG_INNER_BF16), False, 8, 8),
    "b16_naik": (dict(arith=FF, inner=B.STAG_INNER_BF16), True, 8, 8),
    "links16": (dict(arith=FF, inner=B.STAG_INNER_F32_L16), False, 24, 11),
    "links16_naik": (dict(arith=FF, inner=B.STAG_INNER_F32_L16), True, 24, 11),
    "f32_f64": (dict(arith=F64, inner=B.STAG_INNER_F32), True, 24, 24),
}
# V/2 = 1440, 9744, 37800, 75600, 147456
SIZES = [(10, 6, 4, 12), (14, 12, 4, 58), (14, 18, 10, 30), (20, 18, 14, 30), (24, 24, 16, 32)]


def _handle(fat, lng, dims, mass, **kw):
    opt = B.stag_default_options()
    for k, v in kw.items():
        setattr(opt, k, v)
    return B.Handle(torch.from_numpy(fat).cuda(), dims, mass,
                    naik_long=None if lng is None else torch.from_numpy(lng).cuda(), options=opt)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("dims", SIZES, ids=lambda d: "x".join(map(str, d)))
def test_iterates_in_one_launch_and_in_launches(dims, form):
    kw, naik, vec_bits, link_bits = FORMS[form]
    if naik:
        fat, lng = inputs.asqtad_form_fields(dims, seeds=(41, 42, 43))
    else:
        fat, lng = inputs.gauge_field(dims, 41), None
    b = inputs.gaussian_even_source(dims, 44)
    bd = torch.from_numpy(b).cuda()
    xs, counts = [], []
    with _handle(fat, lng, dims, 0.1, **kw) as h:
        for on in (1, 0):
            B.stag_set_one_launch(h.h, on)
            x = torch.zeros_like(bd)
            n = B.stag_launch_count(h.h)
            code, info = B.stag_cg_solve(h.h, bd, x, 1e-14, 3)
            counts.append(B.stag_launch_count(h.h) - n)
            assert code == B.STAG_ERR_NOT_CONVERGED and info["iters"] == 3
            xs.append(x.cpu().numpy().reshape(-1))
    if not (form == "ff_rows" and dims == SIZES[-1]):  # too large for a thread a site
        assert counts[0] < counts[1]
    ref = oracle.cg_fig1(oracle.Operator(fat, lng, 0.1, dims).apply_A, b, np.zeros_like(b), 1e-14, 3)[0]
    size = np.linalg.norm(ref)
    assert np.linalg.norm(xs[0] - xs[1]) <= STORED[vec_bits] * size
    assert np.linalg.norm(xs[0] - ref) <= (STORED[vec_bits] + 64 * 2.0 ** -min(vec_bits, link_bits)) * size


@pytest.mark.parametrize("form", ["f64", "ff"])
def test_runs_of_several_launches(form):
    """More iterations than one launch's 512: launches of 512, 500 and 4096 iterations
    (check_interval 1, 100 and 4096) carry r, d, x and the exchange over and give the same
    bits in FP64, and in float-float the same iterations and x up to its folds' rounding."""
    dims, mass = (8, 6, 4, 10), 0.05  # the oracle takes 1218 iterations
    fat = inputs.gauge_field(dims, 45, eps=1.0)
    b = torch.from_numpy(inputs.gaussian_even_source(dims, 46)).cuda()
    xs, its, counts = [], [], []
    for interval in (1, 100, 4096):
        with _handle(fat, None, dims, mass, arith=F64 if form == "f64" else FF, check_interval=interval) as h:
            x = torch.zeros_like(b)
            _, info = B.stag_cg_solve(h.h, b, x, 1e-10, 1300)
            counts.append(B.stag_launch_count(h.h))
        xs.append(x.cpu().numpy())
        its.append(info["iters"])
    assert its[0] > 1024 and its[1:] == [its[0]] * 2
    assert counts[0] == counts[1] == counts[2] + 2  # three launches against one
    for x in xs[1:]:
        if form == "f64":
            assert np.array_equal(x, xs[0])
        else:
            assert np.linalg.norm(x - xs[0]) <= 1e-13 * np.linalg.norm(xs[0])


def test_two_threads_on_two_handles():
    """Two cooperative grids that each fill the GPU, from two threads and on streams of
    their own: every solve gives the bits it gives alone."""
    cases = [("ff", (20, 18, 14, 30), dict(arith=FF)), ("f32", (24, 24, 16, 32), dict(arith=FF, inner=B.STAG_INNER_F32))]
    work, errors = [], []
    for k, (_, dims, kw) in enumerate(cases):
        h = _handle(inputs.gauge_field(dims, 47 + k), None, dims, 0.2, **kw)
        b = torch.from_numpy(inputs.gaussian_even_source(dims, 49 + k)).cuda()
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        B.stag_set_stream(h.h, s)
        want = torch.zeros_like(b)
        torch.cuda.synchronize()
        assert B.stag_cg_solve(h.h, b, want, 1e-10)[0] == B.STAG_OK
        work.append((h, s, b, want, [torch.zeros_like(b) for _ in range(6)]))
    torch.cuda.synchronize()

    def run(item):
        try:
            h, _, b, _, xs = item
            for x in xs:
                assert B.stag_cg_solve(h.h, b, x, 1e-10)[0] == B.STAG_OK
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=run, args=(w,)) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for h, _, _, want, xs in work:
        assert all(torch.equal(x, want) for x in xs)
        h.close()
