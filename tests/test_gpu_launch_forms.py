"""Lattices small enough for the one-launch CG, iterated in launches of four kernels each
(stag_set_one_launch(h, 0), which takes the way of a device that cannot hold the grid at
once): graphs, direct launches, block lengths and timing, guard bands, and solves of every
storage form on small ragged lattices, where the one launch would otherwise run.

Bars as for the same tests of the one launch: graph replay and direct launches give the same
bits, solves a true residual <= 1e-10 and the oracle's solution to 1e-8.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1010_4782_gb300 import binding as B, inputs  # noqa: E402

pytestmark = pytest.mark.gpu
FF, F64 = B.STAG_ARITH_FF, B.STAG_ARITH_F64
ROWS = dict(long_recon=12, long_scale=inputs.NAIK_COEFF)
# name: (options, Naik links)
FORMS = {
    "f64": (dict(arith=F64), True),
    "ff": (dict(arith=FF), True),
    "ff_rows": (dict(arith=FF, **ROWS), True),
    "f32": (dict(arith=FF, inner=B.STAG_INNER_F32), True),
    "f32_rows_fat": (dict(arith=FF, inner=B.STAG_INNER_F32, link_recon=12), False),
    "f32_rows_naik": (dict(arith=FF, inner=B.STAG_INNER_F32, **ROWS), True),
    "f16": (dict(arith=FF, inner=B.STAG_INNER_F16), True),
    "b16": (dict(arith=FF, inner=B.STAG_INNER_BF16), True),
    "f32_links16": (dict(arith=FF, inner=B.STAG_INNER_F32_L16), True),
    "f32_f64": (dict(arith=F64, inner=B.STAG_INNER_F32), True),
}


def _fields(dims, naik, seed):
    if naik:
        return inputs.asqtad_form_fields(dims, seeds=(seed, seed + 1, seed + 2))
    return inputs.gauge_field(dims, seed), None


def _handle(fat, lng, dims, mass, one_launch=0, **kw):
    opt = B.stag_default_options()
    for k, v in kw.items():
        setattr(opt, k, v)
    h = B.Handle(torch.from_numpy(fat).cuda(), dims, mass, naik_long=None if lng is None else torch.from_numpy(lng).cuda(),
                 options=opt)
    B.stag_set_one_launch(h.h, one_launch)
    return h


@pytest.mark.parametrize("arith", [F64, FF])
def test_graphs_interval_and_timing(arith):
    """Graphs against direct launches: the same bits.  Another block length, or timing: the
    same bits in FP64; in float-float the increment is folded into x once per block, so x may
    differ by its rounding (2^-48 of each of the few dozen folds).  Timing counts one launch
    of each kernel per iteration, the d update not after the last."""
    dims, mass = (6, 4, 2, 8), 0.05
    fat, lng = _fields(dims, True, 29)
    b = torch.from_numpy(inputs.gaussian_even_source(dims, 0)).cuda()
    xs, its, launches = [], [], []
    for kw in ({}, {"use_graphs": 0}, {"check_interval": 1}, {"check_interval": 7, "timing": 1}):
        with _handle(fat, lng, dims, mass, arith=arith, **kw) as h:
            x = torch.zeros_like(b)
            code, info = B.stag_cg_solve(h.h, b, x, 1e-10)
            assert code == B.STAG_OK
            launches.append(B.stag_launch_count(h.h))
            stats = [B.stag_kernel_stats(h.h, k) for k in range(4)]
        xs.append(x.cpu().numpy())
        its.append(info["iters"])
    assert len(set(its)) == 1
    assert all(n >= 4 * its[0] for n in launches)  # the kernels, not the one launch
    assert np.array_equal(xs[0], xs[1])
    for other in xs[2:]:
        if arith == F64:
            assert np.array_equal(xs[0], other)
        else:
            assert np.linalg.norm(other - xs[0]) <= 1e-13 * np.linalg.norm(xs[0])
    assert [n for _, n in stats] == [its[0]] * 3 + [its[0] - 1]
    assert all(ms > 0 for ms, _ in stats)


@pytest.mark.parametrize("form", FORMS)
def test_solve_between_guard_bands(form):
    """Every storage form on a ragged lattice: the oracle's solution, and no byte changed
    around any buffer."""
    dims, mass = (10, 6, 4, 12), 0.05
    kw, naik = FORMS[form]
    fat, lng = _fields(dims, naik, 91)
    b = inputs.gaussian_even_source(dims, 94)
    op = oracle.Operator(fat, lng, mass, dims)
    ref = oracle.solve(op.apply_A, b, tol=1e-13, max_iter=200000, max_restarts=20)["x"]
    with _handle(fat, lng, dims, mass, guard_bands=1, **kw) as h:
        bd = torch.from_numpy(b).cuda()
        x = torch.zeros_like(bd)
        code, info = B.stag_cg_solve(h.h, bd, x, 1e-10, max_iter=20000)
        launches = B.stag_launch_count(h.h)
        checked, bad = B.stag_check_guards(h.h)
    assert code == B.STAG_OK and info["true_rel_residual"] <= 1e-10, info
    assert launches >= 4 * info["iters"]
    assert checked >= 2 * 4096 * 10 and bad == 0
    got = x.cpu().numpy().reshape(-1)
    assert np.linalg.norm(got - ref) <= 1e-8 * np.linalg.norm(ref)


@pytest.mark.parametrize("form", ["f64", "ff", "f32"])
def test_switching_between_the_two(form):
    """The same handle with the one launch, without and with it again: the first and the
    last solve give the same bits, and each way keeps the other's buffers in order."""
    dims, mass = (8, 6, 4, 10), 0.1
    kw, naik = FORMS[form]
    fat, lng = _fields(dims, naik, 61)
    b = torch.from_numpy(inputs.gaussian_even_source(dims, 62)).cuda()
    xs, counts = [], []
    with _handle(fat, lng, dims, mass, one_launch=1, **kw) as h:
        for on in (1, 0, 1, 0):
            B.stag_set_one_launch(h.h, on)
            x = torch.zeros_like(b)
            n = B.stag_launch_count(h.h)
            code, info = B.stag_cg_solve(h.h, b, x, 1e-10)
            assert code == B.STAG_OK
            xs.append(x.cpu().numpy())
            counts.append(B.stag_launch_count(h.h) - n)
    assert np.array_equal(xs[0], xs[2]) and np.array_equal(xs[1], xs[3])
    assert counts[0] < 4 * info["iters"] <= counts[1]
    assert np.linalg.norm(xs[1] - xs[0]) <= 1e-8 * np.linalg.norm(xs[0])


def test_null_handle():
    assert B.load().stag_set_one_launch(None, 0) == B.STAG_ERR_INVALID_ARG
