"""The network's gradient, layer by layer and path by path, against the exact one in FP64 (the
chain rule on the oracle's layers), on lattices of less than one block, of ragged
blocks, and of more sites than one wave of blocks in every layer.

With d = M(r) - e and L = |A d|^2 / |A e|^2 the field g = A^2 d / |A e|^2 is dL/dconj(M(r)), so
G_l[p, o, i] = sum_x g_l,o conj((T_p psi_l-1,i)) with g_l-1 = (layer l)^dag g_l.

Bounds, of the gradient of one path of a layer, relative to the larger of its norm and the
mean path's: every step from r to G rounds its fields by a few units u at random (sums of up
to 216 products), about a dozen steps in all: 64 u with u = 2^-24 in FP32.  BF16 storage
rounds r, e, the activations and the fields g, eight of them, by at most u = 2^-9 each, so
that the expected error is below 2 u: 16 u.
"""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from oracle import ptnet, staggered as st  # noqa: E402
from paper_1010_4782_gb300 import binding as B, inputs  # noqa: E402

pytestmark = pytest.mark.gpu
CHANS = (1, 8, 8, 1)
MASS = 0.2
BOUND = {B.STAG_ARITH_F32: 64 * 2.0 ** -24, B.STAG_ARITH_BF16: 16 * 2.0 ** -9}


@functools.lru_cache(maxsize=1)
def _exact(dims):
    """(fat, r, e, weights, loss, [gradient of each layer])."""
    fat = inputs.gauge_field(dims, 71)
    r, e = inputs.gaussian_even_source(dims, 73), inputs.gaussian_even_source(dims, 74)
    rng = np.random.default_rng(72)
    ws = [(0.3 * (rng.standard_normal((9, co, ci)) + 1j * rng.standard_normal((9, co, ci)))).astype(np.complex64)
          .astype(np.complex128) for ci, co in zip(CHANS[:-1], CHANS[1:])]
    net = ptnet.PTNet(fat, dims, ws)
    op = oracle.Operator(fat, None, MASS, dims)
    acts = net.activations(r)
    d = st.restrict(acts[-1][0], net.dims, 0) - e.reshape(-1, 3)
    ad, ae = op.apply_A(d), op.apply_A(e)
    scale = np.vdot(ae, ae).real
    g = st.embed(op.apply_A(ad).reshape(-1, 3) / scale, net.dims, 0)[None]
    grads = []
    for l in (2, 1, 0):
        psi = acts[l]
        grads.append(np.stack([np.stack([[np.vdot(t, go) for t in tp] for go in g]) for tp in
                               ([ptnet.transport(net.u, ch, p) for ch in psi] for p in range(9))]))
        if l:
            g = ptnet.layer(net.u, ptnet.adjoint_weights(ws[l]), g)
    return fat, r, e, ws, np.vdot(ad, ad).real / scale, grads[::-1]


@pytest.mark.parametrize("dims,prec", [(d, p) for d in ((2, 2, 2, 4), (6, 4, 2, 8), (10, 6, 4, 12), (16, 16, 16, 34))
                                       for p in (B.STAG_ARITH_F32, B.STAG_ARITH_BF16)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_gradient_of_every_layer_and_path(dims, prec):
    fat, r, e, ws, loss, grads = _exact(dims)
    with B.Handle(torch.from_numpy(fat).cuda(), dims, MASS) as h:
        net = B.stag_ptnet_create(h.h, prec, 1)
        try:
            B.stag_ptnet_set_weights(net, np.concatenate([w.ravel() for w in ws]))
            got_loss, flat = B.stag_ptnet_loss_grad(net, torch.from_numpy(r).cuda(), torch.from_numpy(e).cuda())
        finally:
            B.stag_ptnet_destroy(net)
    bound = BOUND[prec]
    assert abs(got_loss - loss) <= bound * loss
    off = 0
    for l, want in enumerate(grads):
        got = flat[off:off + want.size].reshape(want.shape)
        off += want.size
        mean = np.linalg.norm(want) / 3.0
        for p in range(9):
            err = np.linalg.norm(got[p] - want[p]) / max(np.linalg.norm(want[p]), mean)
            assert err <= bound, (l, p, err)
    assert off == flat.size
