"""The performance cases of the staggered even-odd CG library.

Each case is one call (or one short sequence of calls) that a program using the
library makes through its public binding, with everything such a program keeps
between calls - the handle or batch, the network, the link and source arrays -
prepared beforehand on the GPU.  Lattices, operators, masses and tolerances are
those of the benchmark's workloads and of the test suite: synthetic SU(3) links
exp(0.3 i H), the one-hop operator or the asqtad form (fat 0.6 U_a + 0.4 U_b,
Naik -U_c/24), Gaussian even-site sources, true residual 1e-10.

Kinds:
  solve      stag_cg_solve on a kept handle (one source after another on one field)
  new_field  stag_create_ex + stag_cg_solve + stag_destroy (a field used once, as
             in a gauge-generation program; the benchmark's step)
  apply      stag_apply_A (programs that run their own Krylov or eigenvalue loop)
  batch      stag_batch_solve: many right-hand sides on one field
  lattices   stag_batch_solve: independent fields of different sizes
  fcg        stag_fcg_solve with the network preconditioner
  grad       stag_ptnet_loss_grad: one pair of the network's training
"""
import math

import numpy as np
import torch

from paper_1010_4782_gb300 import binding as B

TOL = 1e-10
EPS = 0.3
NAIK = -1.0 / 24.0
AXIS = (3, 2, 1, 0)  # direction x, y, z, t -> axis of a [Lt, Lz, Ly, Lx] array
HIDDEN = 8
PATHS = 9

# arithmetic forms: (arith, inner, link_recon, long_recon)
FORMS = {
    "f64": (B.STAG_ARITH_F64, B.STAG_INNER_NONE, 0, 0),
    "ff": (B.STAG_ARITH_FF, B.STAG_INNER_NONE, 0, 0),
    "f32": (B.STAG_ARITH_FF, B.STAG_INNER_F32, 0, 0),
    "f32_rows_fat": (B.STAG_ARITH_FF, B.STAG_INNER_F32, 12, 0),
    "f32_rows_naik": (B.STAG_ARITH_FF, B.STAG_INNER_F32, 0, 12),
    "f16": (B.STAG_ARITH_FF, B.STAG_INNER_F16, 0, 0),
    "f32_links16": (B.STAG_ARITH_FF, B.STAG_INNER_F32_L16, 0, 0),
}
# bytes of a real number in the iteration's links and vectors
REAL_BYTES = {"f64": (8, 8), "ff": (8, 8), "f32": (4, 4), "f32_rows_fat": (4, 4), "f32_rows_naik": (4, 4),
              "f16": (2, 2), "f32_links16": (2, 4)}


def _case(kind, dims, naik, form="ff", mass=0.031, rhs=1, name=None):
    c = {"kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3], "naik": bool(naik), "form": form,
         "mass": float(mass), "rhs": int(rhs)}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest system anyone solves: a test lattice, plain FP64
        _case("solve", (4, 4, 4, 4), False, "f64", 0.1, name="solve_f64_4x4x4x4"),
        # a small production-like lattice in the default FP64-class arithmetic
        _case("solve", (8, 8, 8, 16), True, "ff", 0.05, name="solve_ff_8x8x8x16"),
        # an ordinary lattice with ragged extents (V/2 not a multiple of 64), mixed precision
        _case("solve", (20, 18, 14, 30), True, "f32", 0.031, name="solve_f32_20x18x14x30"),
        # the paper's lattice at the workload's second mass: plain CG, FP64 class
        _case("solve", (28, 28, 28, 96), True, "ff", 0.031, name="solve_ff_28x28x28x96"),
        # the same system in the fastest form that holds at every mass
        _case("solve", (28, 28, 28, 96), True, "f32_rows_naik", 0.031, name="solve_rows_28x28x28x96"),
        # and with FP16 links and vectors, the fastest at this mass
        _case("solve", (28, 28, 28, 96), True, "f16", 0.031, name="solve_f16_28x28x28x96"),
        # a field that is packed, solved on once and dropped (12-parameter links)
        _case("new_field", (24, 24, 24, 48), False, "f32_rows_fat", 0.05, name="new_field_24x24x24x48"),
        # one application of A inside a caller's own iteration
        _case("apply", (32, 32, 32, 64), True, "ff", 0.0062, name="apply_ff_32x32x32x64"),
        # propagator production: 16 right-hand sides on one field
        _case("batch", (24, 24, 24, 48), True, "f32", 0.05, 16, name="batch_16_24x24x24x48"),
        # independent lattices of three sizes in one batch (8^4, 16^4 and 24^3 x 48)
        _case("lattices", (24, 24, 24, 48), False, "f32", 0.05, 10, name="lattices_10"),
        # flexible CG with the network
        _case("fcg", (24, 24, 24, 48), True, "ff", 0.031, name="fcg_24x24x24x48"),
        # one training pair of the network
        _case("grad", (16, 16, 16, 32), True, "ff", 0.0062, name="grad_16x16x16x32"),
    ]


# Largest V/2 (times right-hand sides for a batch) that a drawn case takes: each
# costs no more than the largest listed case.
_CAP = {"f64": 80_000, "ff": 900_000, "f32": 1_000_000, "f32_rows_fat": 1_000_000, "f32_rows_naik": 1_000_000,
        "f16": 1_000_000, "f32_links16": 1_000_000}


def _extents(rng, lo, hi):
    """Even extents with V/2 between lo and hi, spread over the logarithm."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        stretch = math.exp(rng.uniform(0.0, math.log(4.0)))
        side = (2.0 * target / stretch) ** 0.25
        d = [max(4, 2 * round(side * math.exp(rng.uniform(-0.25, 0.25)) / 2)) for _ in range(3)]
        d.append(max(4, 2 * round(side * stretch / 2)))
        if 0.5 * lo <= d[0] * d[1] * d[2] * d[3] // 2 <= hi:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["solve"] * 5 + ["new_field", "apply", "batch", "lattices", "fcg", "grad"])
    mass = round(math.exp(rng.uniform(math.log(0.031), math.log(0.1))), 4)
    naik = rng.random() < 0.6
    if kind in ("solve", "new_field"):
        form = rng.choice(["f64", "ff", "f32", "f16", "f32_links16", "f32_rows_naik" if naik else "f32_rows_fat"])
        if form in ("f16", "f32_links16"):
            mass = max(mass, 0.05)  # FP16-rounded links need m^2 well above their rounding
        return _case(kind, _extents(rng, 128, _CAP[form]), naik, form, mass)
    if kind == "apply":
        form = rng.choice(["f64", "ff"])
        return _case(kind, _extents(rng, 128, 1_000_000), naik, form, mass)
    if kind == "batch":
        rhs = rng.randint(2, 16)
        return _case(kind, _extents(rng, 1024, 300_000 * 16 // max(rhs, 16)), naik, "f32", max(mass, 0.05), rhs)
    if kind == "lattices":
        return _case(kind, _extents(rng, 8192, 300_000), naik, "f32", max(mass, 0.05), rng.randint(3, 10))
    if kind == "fcg":
        return _case(kind, _extents(rng, 2048, 300_000), True, rng.choice(["ff", "ff", "f64"]) if mass > 0.05 else "ff",
                     mass)
    return _case("grad", _extents(rng, 2048, 80_000), naik, "ff", mass)


# ------------------------------------------------------------------ inputs
def _dims(c):
    return c["lx"], c["ly"], c["lz"], c["lt"]


def _half(dims):
    return dims[0] * dims[1] * dims[2] * dims[3] // 2


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(shape, gen):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device="cuda", dtype=torch.float64))


def _mul3(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _su3(dims, gen):
    """Links exp(0.3 i H), H Gaussian Hermitian traceless, as [Lt, Lz, Ly, Lx, 4, 3, 3]."""
    lx, ly, lz, lt = dims
    n = 8 * _half(dims)
    out = torch.empty(n, 3, 3, dtype=torch.complex128, device="cuda")
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    for s in range(0, n, 1 << 20):
        e = min(n, s + (1 << 20))
        m = _normal((e - s, 3, 3), gen)
        h = 0.5 * (m + m.mH)
        h = h - (torch.diagonal(h, dim1=-2, dim2=-1).sum(-1).real / 3.0)[:, None, None] * eye
        a = (0.25j * EPS) * h  # exp(a)^4: a Taylor series of the quarter, then two squarings
        u = eye + a / 14.0
        for k in range(13, 0, -1):
            u = eye + _mul3(a, u) / k
        u = _mul3(u, u)
        out[s:e] = _mul3(u, u)
    return out.view(lt, lz, ly, lx, 4, 3, 3)


def _fields(dims, naik, seed):
    """(fat, Naik or None): the asqtad form, or SU(3) one-hop links."""
    gen = _generator(seed)
    fat = _su3(dims, gen)
    if not naik:
        return fat, None
    fat = 0.6 * fat + 0.4 * _su3(dims, gen)
    return fat, NAIK * _su3(dims, gen)


def _source(dims, seed):
    return _normal((_half(dims), 3), _generator(seed))


def _options(form):
    o = B.stag_default_options()
    o.arith, o.inner, o.link_recon, o.long_recon = FORMS[form]
    if o.long_recon:
        o.long_scale = NAIK
    return o


def _lattice_sizes(c):
    """The extents of a batch of independent lattices: 8^4, 16^4 and the case's own size
    in turn (twice each of the small ones for one of the large)."""
    own = _dims(c)
    cycle = [(8, 8, 8, 8), (16, 16, 16, 16), (8, 8, 8, 8), own, (16, 16, 16, 16)]
    return [cycle[k % 5] for k in range(c["rhs"])]


def _lattice_masses(c):
    n = c["rhs"]
    return [c["mass"] * (0.5 + 0.5 * k / max(1, n - 1)) for k in range(n)]


def _weights(seed, mass):
    """Network weights near its polynomial start (M r ~ alpha r + beta A r in the
    self-adjoint form), with the spread that training leaves."""
    rng = np.random.default_rng(seed)
    w = [0.01 * (rng.standard_normal((PATHS, o, i)) + 1j * rng.standard_normal((PATHS, o, i)))
         for o, i in ((HIDDEN, 1), (HIDDEN, HIDDEN), (1, HIDDEN))]
    lmax = 16.0
    alpha, beta = 4.0 / lmax, -10.0 / (3.0 * lmax * lmax)
    w[0][0, 0, 0] += 1.0
    w[1][0, 0, 0] += alpha + beta * mass * mass
    w[1][0, 1, 1] += beta
    w[2][0, 0, 0] += 1.0
    for mu in range(4):
        w[0][1 + 2 * mu, 1, 0] += 1.0
        w[0][2 + 2 * mu, 1, 0] -= 1.0
        w[2][1 + 2 * mu, 0, 1] -= 1.0
        w[2][2 + 2 * mu, 0, 1] += 1.0
    # the library keeps its weights in FP32
    return [x.astype(np.complex64).astype(np.complex128) for x in w]


class _Batch:
    def __init__(self, *args):
        self.h = B.stag_batch_create(*args)

    def __del__(self):
        B.stag_batch_destroy(self.h)


class _Net:
    def __init__(self, handle, seed):
        self.handle = handle  # the network points at it: kept alive, destroyed after
        self.n = B.stag_ptnet_create(handle.h, B.STAG_ARITH_BF16, seed)

    def __del__(self):
        B.stag_ptnet_destroy(self.n)


def _pair(apply_a, dims, seed):
    """A training pair: e a vector with its rough modes damped, r = A e, both over |r|."""
    e = _source(dims, seed)
    for _ in range(4):
        e = e - apply_a(e) / 20.0
    r = apply_a(e)
    n = torch.linalg.vector_norm(r)
    return r / n, e / n


def prepare(case, seed):
    kind, dims, mass = case["kind"], _dims(case), case["mass"]
    s = {"kind": kind, "dims": dims, "mass": mass}
    if kind == "lattices":
        sizes, masses = _lattice_sizes(case), _lattice_masses(case)
        fields = [_fields(d, case["naik"], seed + 1000 * k) for k, d in enumerate(sizes)]
        s["b"] = [_source(d, seed + 1000 * k + 500) for k, d in enumerate(sizes)]
        s["x"] = [torch.zeros_like(b) for b in s["b"]]
        s["batch"] = _Batch([f for f, _ in fields], [l for _, l in fields], sizes, masses)
        return s
    fat, lng = _fields(dims, case["naik"], seed)
    if kind == "batch":
        n = case["rhs"]
        s["b"] = [_source(dims, seed + 1 + k) for k in range(n)]
        s["x"] = [torch.zeros_like(b) for b in s["b"]]
        s["batch"] = _Batch([fat] * n, [lng] * n, [dims] * n, [mass] * n)
        return s
    if kind == "new_field":
        s.update(fat=fat, lng=lng, opt=_options(case["form"]))
    else:
        s["h"] = B.Handle(fat, dims, mass, naik_long=lng, options=_options(case["form"]))
    s["b"] = _source(dims, seed + 1)
    s["x"] = torch.zeros_like(s["b"])
    if kind == "fcg":
        s["net"] = _Net(s["h"], 1)
    elif kind == "grad":
        s["net"] = _Net(s["h"], 1)
        B.stag_ptnet_set_weights(s["net"].n, np.concatenate([w.ravel() for w in _weights(seed, mass)]))

        def apply_a(v):
            out = torch.empty_like(v)
            B.stag_apply_A(s["h"].h, v.contiguous(), out)
            return out

        s["r"], s["e"] = _pair(apply_a, dims, seed + 1)
    return s


# --------------------------------------------------------------------- run
def run(s):
    kind = s["kind"]
    if kind == "solve":
        s["x"].zero_()
        B.stag_cg_solve(s["h"].h, s["b"], s["x"], TOL)
        return s["x"]
    if kind == "new_field":
        s["x"].zero_()
        with B.Handle(s["fat"], s["dims"], s["mass"], naik_long=s["lng"], options=s["opt"]) as h:
            B.stag_cg_solve(h.h, s["b"], s["x"], TOL)
        return s["x"]
    if kind == "apply":
        B.stag_apply_A(s["h"].h, s["b"], s["x"])
        return s["x"]
    if kind in ("batch", "lattices"):
        for x in s["x"]:
            x.zero_()
        B.stag_batch_solve(s["batch"].h, s["b"], s["x"], TOL)
        return s["x"]
    if kind == "fcg":
        s["x"].zero_()
        B.stag_fcg_solve(s["h"].h, s["net"].n, s["b"], s["x"], TOL)
        return s["x"]
    loss, grad = B.stag_ptnet_loss_grad(s["net"].n, s["r"], s["e"])
    # the network's gradients are sums of FP32 numbers: an optimiser keeps them in FP32
    return {"loss": np.float32(loss), "grad": grad.astype(np.complex64)}


# -------------------------------------------------------------------- work
def _iterations(mass):
    """CG iterations to 1e-10: about 20.6 / m on these fields (666 at m = 0.031)."""
    return 20.6 / mass


def _cg_work(dims, naik, form, mass, rhs=1):
    """CG with the links and the CG vectors in the iteration's storage: per iteration each
    link once, x, r, d and A d once each way; 72 flops a hop, two half-Dslashes."""
    vh, hops = _half(dims), 16 if naik else 8
    lb, vb = REAL_BYTES[form]
    fat = 8 * (6 if form == "f32_rows_fat" else 9) * 2 * lb
    lng = 8 * (6 if form == "f32_rows_naik" else 9) * 2 * lb if naik else 0
    n = _iterations(mass)
    return n * vh * (fat + lng + rhs * 8 * 6 * vb), n * vh * rhs * (2 * hops * 72 + 60)


def work(case):
    kind, dims, naik, mass = case["kind"], _dims(case), case["naik"], case["mass"]
    vh, hops = _half(dims), 16 if naik else 8
    links = 2 * 4 * 9 * 16 * vh * (2 if naik else 1)  # the caller's complex128 links
    if kind == "apply":
        return {"bytes": links + 2 * 48 * vh, "flops": vh * (2 * hops * 72 + 12)}
    if kind == "lattices":
        each = [_cg_work(d, naik, "f32", m) for d, m in zip(_lattice_sizes(case), _lattice_masses(case))]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    if kind == "grad":
        # the links and the pair once; forward, adjoint and weight gradient of the 8 -> 8
        # layer (8 transports of 8 channels, 9 x 64 complex weights on 3 colours) on every
        # site, and three applications of A
        site = 3 * (8 * 8 * 72 + 9 * 64 * 3 * 8)
        return {"bytes": links + 2 * 48 * vh, "flops": 2 * vh * site + 3 * vh * 2 * hops * 72}
    b, f = _cg_work(dims, naik, case["form"], mass, case["rhs"])
    if kind == "fcg":  # about two thirds of the iterations, each with 16 one-hop transports more
        b, f = 0.67 * (b + _iterations(mass) * vh * 8 * 18 * 2), 0.67 * (f + _iterations(mass) * vh * (16 * 72 + 512 * 3))
    if kind == "new_field":
        b += links
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------- exact
class _Operator:
    """A = m^2 - D_eo D_oe on even sites, plain torch in 64 bits (whole-lattice arrays)."""

    def __init__(self, fat, lng, dims, mass):
        lx, ly, lz, lt = dims
        t, z, y, x = torch.meshgrid(*(torch.arange(n, device="cuda") for n in (lt, lz, ly, lx)), indexing="ij")
        self.dims, self.m2 = dims, mass * mass
        self.even = ((x + y + z + t) % 2 == 0).reshape(-1).nonzero().reshape(-1)
        phase = [torch.zeros_like(x), x, x + y, x + y + z]
        self.hops = []  # (matrix, direction, shift) of +U v(x + h mu) - U(x - h mu)^dag v(x - h mu)
        self.fat = []
        for links, h in ((fat, 1), (lng, 3)):
            if links is None:
                continue
            for mu in range(4):
                u = links[..., mu, :, :] * (1.0 - 2.0 * (phase[mu] % 2)).to(links.dtype)[..., None, None]
                back = torch.roll(u, h, AXIS[mu]).mH.contiguous()
                self.hops += [(u, mu, h, 1.0), (back, mu, -h, -1.0)]
                if h == 1:
                    self.fat += [(u, mu, 1), (back, mu, -1)]

    def transport(self, k, v):
        """Path k + 1 of the network: U v from x + mu, or U^dag v from x - mu; v [..., C, 3]."""
        u, mu, h = self.fat[k]
        return (u.unsqueeze(-3) * torch.roll(v, -h, AXIS[mu]).unsqueeze(-2)).sum(-1)

    def embed(self, v):
        lx, ly, lz, lt = self.dims
        f = torch.zeros(lt * lz * ly * lx, 3, dtype=torch.complex128, device="cuda")
        f = f.index_copy(0, self.even, v)
        return f.view(lt, lz, ly, lx, 3)

    def restrict(self, f):
        return f.reshape(-1, 3)[self.even]

    def dslash(self, f):
        out = torch.zeros_like(f)
        for u, mu, h, sign in self.hops:
            out = out + sign * (u * torch.roll(f, -h, AXIS[mu]).unsqueeze(-2)).sum(-1)
        return out

    def __call__(self, v):
        return self.m2 * v - self.restrict(self.dslash(self.dslash(self.embed(v))))


def _solve(op, b, tol=1e-13, most=4000):
    x, r = torch.zeros_like(b), b.clone()
    d, rr = r.clone(), torch.vdot(r.view(-1), r.view(-1)).real
    stop = tol * tol * float(rr)
    for _ in range(most):
        ad = op(d)
        alpha = rr / torch.vdot(d.view(-1), ad.view(-1)).real
        x += alpha * d
        r -= alpha * ad
        new = torch.vdot(r.view(-1), r.view(-1)).real
        d = r + (new / rr) * d
        rr = new
        if float(rr) <= stop:
            break
    return x


def exact(case, seed):
    kind, dims, mass = case["kind"], _dims(case), case["mass"]
    if kind == "lattices":
        out, seen = [], set()
        for k, (d, m) in enumerate(zip(_lattice_sizes(case), _lattice_masses(case))):
            if d in seen:  # one system of each size
                out.append(None)
                continue
            seen.add(d)
            fat, lng = _fields(d, case["naik"], seed + 1000 * k)
            out.append(_solve(_Operator(fat, lng, d, m), _source(d, seed + 1000 * k + 500)))
        return out
    fat, lng = _fields(dims, case["naik"], seed)
    op = _Operator(fat, lng, dims, mass)
    if kind == "batch":  # the first four right-hand sides
        return [_solve(op, _source(dims, seed + 1 + k)) if k < 4 else None for k in range(case["rhs"])]
    if kind == "apply":
        return op(_source(dims, seed + 1))
    if kind == "grad":
        r, e = _pair(op, dims, seed + 1)
        w = [torch.from_numpy(x).cuda().requires_grad_() for x in _weights(seed, mass)]
        psi = op.embed(r).unsqueeze(-2)
        for l in range(3):
            out = torch.einsum("oi,...ic->...oc", w[l][0], psi)
            for k in range(PATHS - 1):
                out = out + torch.einsum("oi,...ic->...oc", w[l][k + 1], op.transport(k, psi))
            psi = out
        ad, ae = op(op.restrict(psi.squeeze(-2)) - e), op(e)
        loss = ad.abs().square().sum() / ae.abs().square().sum()
        g = torch.autograd.grad(loss, w)
        # torch gives dL/dRe + i dL/dIm = 2 dL/d conj(W)
        return {"loss": loss.detach(), "grad": torch.cat([0.5 * x.reshape(-1) for x in g])}
    return _solve(op, _source(dims, seed + 1))
