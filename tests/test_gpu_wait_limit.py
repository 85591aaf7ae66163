"""A wait between the blocks of the one-launch CG that runs out (here after 0 to 3 polls
instead of two seconds): the call returns STAG_ERR_TIMEOUT and leaves x as it was, and the
handle's next solves give the bits of the solve before it, whatever exchange each block
had left at.  With no polls every block but the last to arrive gives up, so the error
is certain; with one to three some launches get through some exchanges first."""
import pytest

torch = pytest.importorskip("torch")
from paper_1010_4782_gb300 import binding, inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["f64", "ff", "f32"])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 6, 4, 10), (14, 18, 10, 30)],
                         ids=lambda d: "x".join(map(str, d)))
def test_solves_after_a_wait_ran_out(dims, form):
    opt = binding.stag_default_options()
    opt.arith = binding.STAG_ARITH_F64 if form == "f64" else binding.STAG_ARITH_FF
    opt.inner = binding.STAG_INNER_F32 if form == "f32" else binding.STAG_INNER_NONE
    opt.timing = 1
    fat = torch.from_numpy(inputs.gauge_field(dims, 51)).cuda()
    b = torch.from_numpy(inputs.gaussian_even_source(dims, 52)).cuda()
    with binding.Handle(fat, dims, 0.3, options=opt) as h:
        want = torch.zeros_like(b)
        assert binding.stag_cg_solve(h.h, b, want, 1e-10)[0] == binding.STAG_OK
        for limit in (0, 1, 2, 3, 0):
            binding.stag_set_wait_limit(h.h, limit)
            x = torch.zeros_like(b)
            code, _ = binding.stag_cg_solve(h.h, b, x, 1e-10, raise_on_error=False)
            if limit == 0:
                assert code == binding.STAG_ERR_TIMEOUT and "wait" in binding.stag_last_error(h.h)
            if code == binding.STAG_ERR_TIMEOUT:
                assert not x.any()
            else:
                assert torch.equal(x, want)
            binding.stag_set_wait_limit(h.h, -1)
            binding.stag_reset_stats(h.h)
            for _ in range(2):
                x.zero_()
                code, info = binding.stag_cg_solve(h.h, b, x, 1e-10)
                assert code == binding.STAG_OK and torch.equal(x, want)
            assert binding.stag_kernel_stats(h.h, 0)[1] == 2 * info["iters"]


def test_null_handle():
    assert binding.load().stag_set_wait_limit(None, 0) == binding.STAG_ERR_INVALID_ARG
