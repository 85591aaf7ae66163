"""The network's weight-gradient kernels at the edges of their grids, against the loss
itself (no oracle: a directional derivative of a quadratic)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1010_4782_gb300 import binding, inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (6, 4, 2, 8), (10, 6, 4, 12), (12, 12, 12, 26)],
                         ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("prec", [binding.STAG_ARITH_F32, binding.STAG_ARITH_BF16])
def test_weight_gradient_grids(dims, prec):
    """The weight gradient on lattices of less than one block, ragged blocks and more sites
    than one wave of blocks: the sum of G conj(dW) over a random direction dW equals the
    directional derivative of the loss, which for a linear network and a quadratic loss
    is exact from the two end points.  Bounds: the FP32 sums of the gradient and of the
    loss (2^-24 times a few hundred rounded terms), and BF16 activations (2^-9 each, of
    three layers and their adjoints)."""
    fat = inputs.gauge_field(dims, 71)
    rng = np.random.default_rng(72)
    w = 0.3 * (rng.standard_normal(720) + 1j * rng.standard_normal(720))
    dw = rng.standard_normal(720) + 1j * rng.standard_normal(720)
    dw[:72] = 0.0   # second layer only: the loss is then quadratic in the step
    dw[72 + 576:] = 0.0
    r = torch.from_numpy(inputs.gaussian_even_source(dims, 73)).cuda()
    e = torch.from_numpy(inputs.gaussian_even_source(dims, 74)).cuda()
    with binding.Handle(torch.from_numpy(fat).cuda(), dims, 0.2) as h:
        net = binding.stag_ptnet_create(h.h, prec, 1)
        try:
            assert w.size == binding.stag_ptnet_weights(net).size
            binding.stag_ptnet_set_weights(net, w)
            _, g = binding.stag_ptnet_loss_grad(net, r, e)
            ends = []
            for s in (1.0, -1.0):
                binding.stag_ptnet_set_weights(net, w + s * dw)
                ends.append(binding.stag_ptnet_loss_grad(net, r, e)[0])
        finally:
            binding.stag_ptnet_destroy(net)
    want = 0.5 * (ends[0] - ends[1])           # dL along dw, exact for a quadratic
    got = 2.0 * np.real(np.vdot(g, dw))        # dL = 2 Re sum conj(G) dW
    scale = 2.0 * np.linalg.norm(g) * np.linalg.norm(dw) / np.sqrt(dw.size) + abs(want)
    bound = 1e-4 if prec == binding.STAG_ARITH_F32 else 3 * 6 * 2.0 ** -9
    assert abs(got - want) <= bound * (scale + ends[0] + ends[1])
