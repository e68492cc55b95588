"""Performance cases: the work that users of the library have it do, through ``pd.Plan``, ``pd.Batch`` and
``autograd``, with the plans' built-in pass configuration, from one force evaluation on a small 2D grid to the
largest 3D box, the solvers and the dynamic drivers.

A case is a dict of plain values. ``kind`` picks the entry point:

  force     L (and W) = Plan.force(u): the operator itself, bond (2D / 3D), state-based or nonlinear model
  grad      autograd.pd_force with a node weight s, forward and backward (L, dJ/du, dJ/ds)
  dynamics  Plan.step_verlet from a saved state (u, v, lambda after the steps)
  static    Plan.solve_static from u = 0
  relax     Batch.solve_dr: uneven 2D specimens in one graph launch
  inverse   autograd.verlet_loss and its gradient with respect to the micromodulus

``n`` are the grid lengths x1, x2[, x3] ("128x128x64"), ``fill`` the part of the box that the body takes along
each axis (bodies are padded up to power-of-two boxes, so the far side of the box is empty in earnest).
"""
import math

import numpy as np
import torch

from paper_2105_06055_gb300 import autograd, pd

DEV = "cuda"


# ---------------------------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one evaluation on a 128 x 128 plate in double precision, as in a step of a user's
        # own time stepping or parameter study; launches and latency count
        dict(name="force 2d 128 f64", kind="force", n="128x128", fp64=True, delta=3.0, fill=0.8),
        # a plate of the fracture workload's size, force and energy density of a linearized bond model
        dict(name="force+energy 2d 1024x512", kind="force", n="1024x512", delta=4.0, fill=1.0, energy=True),
        # the scale sweep of one 3D force evaluation (bond model): 128^3, 256^3 and the largest box, 512^3
        dict(name="force 3d 128", kind="force", n="128x128x128", delta=3.0, fill=1.0),
        dict(name="force 3d 256", kind="force", n="256x256x256", delta=3.0, fill=1.0),
        dict(name="force 3d 512", kind="force", n="512x512x512", delta=3.0, fill=1.0),
        # the state-based solid with dilatation (nu = 0.4), on a box whose lengths differ
        dict(name="state 3d 256x128x128", kind="force", n="256x128x128", model="state", delta=3.0, fill=0.9),
        # the nonlinear rotation-invariant bond model: the widest passes (12 forward, 21 inverse fields)
        dict(name="nonlinear 3d 64x64x64", kind="force", n="64x64x64", model="nonlinear", delta=2.5, fill=1.0),
        # training-style use: weighted force through torch autograd, forward and backward
        dict(name="grad 3d 128", kind="grad", n="128x128x128", delta=3.0, fill=1.0),
        # dynamic fracture, the 1024 x 512 notched plate in single precision with the horizon-sum energy
        dict(name="dynamics 2d 1024x512", kind="dynamics", n="1024x512", delta=4.0, fill=1.0, steps=20, load=0.3),
        # the elastostatic solve (cube minus a ball, clamp and load layers, state-based nu = 0.25): FP32 conjugate
        # gradients with FP64 refinement, to a residual that leaves nine digits of the displacement
        dict(name="static 3d 128", kind="static", n="128x128x128", delta=3.0, fill=1.0, rtol=1e-10),
        # a batch of uneven specimens (sides 40 to 128 padded to powers of two) by dynamic relaxation, which leaves
        # more of the residual in the lowest modes than conjugate gradients: one digit further
        dict(name="relax 2d batch", kind="relax", n="128x128", delta=4.0, count=6, rtol=1e-11),
        # the inverse problem: dynamics with a variable micromodulus, loss and gradient, double precision
        dict(name="inverse 3d 64 f64", kind="inverse", n="64x64x64", fp64=True, delta=3.0, fill=1.0, steps=8),
    ]


def draw(rng):
    kind = rng.choice(["force", "force", "force", "grad", "dynamics", "static", "relax", "inverse"])
    p2 = lambda lo, hi: 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))  # noqa: E731
    x = lambda *n: "x".join(str(v) for v in n)  # noqa: E731
    fill = round(rng.uniform(0.55, 1.0), 3)
    if kind == "force":
        form = rng.choice(["bond2", "bond2", "bond3", "bond3", "state", "nonlinear"])
        if form == "bond2":
            fp64 = rng.random() < 0.4
            top = 512 if fp64 else 1024
            return dict(kind=kind, n=x(p2(64, 2 * top), p2(64, top)), fp64=fp64, fill=fill,
                        delta=round(rng.uniform(2.0, 5.0), 2), energy=rng.random() < 0.4)
        if form == "bond3":
            fp64 = rng.random() < 0.25
            top = 128 if fp64 else 512
            return dict(kind=kind, n=x(p2(32, top), p2(32, top), p2(32, top)), fp64=fp64, fill=fill,
                        delta=round(rng.uniform(2.0, 4.0), 2))
        top = 256 if form == "state" else 128
        return dict(kind=kind, n=x(p2(32, top), p2(32, top), p2(32, top)), model=form, fill=fill,
                    delta=round(rng.uniform(2.0, 3.5), 2))
    if kind == "grad":
        if rng.random() < 0.4:
            return dict(kind=kind, n=x(p2(64, 1024), p2(64, 512)), delta=round(rng.uniform(2.0, 5.0), 2), fill=fill)
        return dict(kind=kind, n=x(p2(32, 128), p2(32, 128), p2(32, 128)), delta=round(rng.uniform(2.0, 3.5), 2),
                    fill=fill)
    if kind == "dynamics":
        # in double precision also through the breaking of bonds at the notch's tip (load > 1)
        fp64 = rng.random() < 0.5
        return dict(kind=kind, n=x(p2(128, 1024), p2(128, 512)), fp64=fp64, delta=float(rng.randint(3, 5)),
                    fill=1.0, steps=rng.randint(5, 30), load=1.6 if fp64 else 0.3)
    if kind == "static":
        return dict(kind=kind, n=x(p2(32, 128), p2(32, 128), p2(32, 128)), delta=round(rng.uniform(2.0, 3.5), 2),
                    fill=fill, rtol=1e-10)
    if kind == "relax":
        return dict(kind=kind, n="128x128", delta=float(rng.randint(3, 5)), count=rng.randint(2, 6), rtol=1e-11)
    return dict(kind=kind, n=x(p2(32, 64), p2(32, 64), p2(32, 64)), fp64=True, delta=round(rng.uniform(2.0, 3.0), 2),
                fill=fill, steps=rng.randint(4, 10))


# ---------------------------------------------------------------------------------------------------------------
# Inputs, made on the GPU from the seed
# ---------------------------------------------------------------------------------------------------------------

def _shape(case):
    """C-order shape, x1 last."""
    return tuple(int(v) for v in case["n"].split("x"))[::-1]


def _dtype(case):
    return torch.float64 if case.get("fp64") else torch.float32


def _axis(shape, a, dtype=torch.float64):
    """Node indices along x_(a+1), shaped to broadcast over the grid."""
    d = len(shape)
    v = [1] * d
    v[d - 1 - a] = shape[d - 1 - a]
    return torch.arange(shape[d - 1 - a], device=DEV, dtype=dtype).view(v)


def _body(case, g, hole=True):
    """A box delta away from the faces, ``fill`` of the free length along each axis, minus an off-centre
    ellipsoid. Returns the mask (bool) and the body's extent along x1."""
    shape = _shape(case)
    d = len(shape)
    m = int(math.ceil(case["delta"]))
    chi = torch.ones(shape, dtype=torch.bool, device=DEV)
    r2 = torch.zeros((1,) * d, device=DEV, dtype=torch.float64)
    ext = []
    for a in range(d):
        n = shape[d - 1 - a]
        hi = max(m + 2 * m + 4, m + int(round(case.get("fill", 1.0) * (n - 2 * m))))
        hi = min(hi, n - m)
        ext.append((m, hi))
        i = _axis(shape, a)
        chi &= (i >= m) & (i < hi)
        c, r = m + g.uniform(0.42, 0.58) * (hi - m), g.uniform(0.15, 0.27) * (hi - m)
        r2 = r2 + ((i - c) / r) ** 2
    if hole:
        chi &= r2 >= 1.0
    return chi, ext


def _waves(shape, ncomp, g, amp, terms=3, short=12.0, long=48.0):
    """Smooth fields: per component a sum of products of sine waves, wave lengths of 12 to 48 nodes."""
    d = len(shape)
    out = torch.zeros((ncomp,) + shape, dtype=torch.float64, device=DEV)
    for c in range(ncomp):
        for _ in range(terms):
            f = torch.full((1,) * d, amp / terms, device=DEV, dtype=torch.float64)
            for a in range(d):
                n = shape[d - 1 - a]
                k = int(g.integers(max(1, int(n / long)), max(2, int(n / short) + 1)))
                f = f * torch.sin(2 * math.pi * k / n * _axis(shape, a) + g.uniform(0, 2 * math.pi))
            out[c] += f
    return out


def _model(case):
    return {"bond": pd.PD_LIN_BOND, "state": pd.PD_LIN_STATE, "nonlinear": pd.PD_NONLIN_BOND}[case.get("model", "bond")]


def _problem(case, **more):
    return pd.Problem(shape=_shape(case), delta=case["delta"], model=_model(case), fp64=bool(case.get("fp64")),
                      **more)


def _clamped(chi, ext, case, g):
    """Clamp on the delta layers at the x1-low face, body force on those at the x1-high face, in a seeded direction."""
    shape = _shape(case)
    d = len(shape)
    w = int(math.ceil(case["delta"]))
    i = _axis(shape, 0)
    om = chi & (i >= ext[0][0] + w)
    layer = (chi & (i >= ext[0][1] - w)).double()
    t = g.normal(size=d)
    t[0] = abs(t[0]) + 1.0
    t *= 1e-3 / case["delta"] / np.linalg.norm(t)
    b = torch.stack([layer * float(v) for v in t])
    return om, b


def _notch(case, chi):
    """Integrity of the plate with a delta-thick notch along the middle, and the tip's place."""
    shape = _shape(case)
    n2, n1 = shape
    delta, m = case["delta"], int(math.ceil(case["delta"]))
    tip, mid = m + (n1 - 2 * m) // 2, n2 / 2.0 - 0.5
    x1, x2 = _axis(shape, 0), _axis(shape, 1)
    cut = (x1 < tip) & ((x2 - mid).abs() < delta / 2.0)
    return chi & ~cut, tip, mid


def _inputs(case, seed):
    """The tensors of a case (without plans)."""
    g = np.random.Generator(np.random.PCG64(int(seed)))
    shape, dt, kind = _shape(case), _dtype(case), case["kind"]
    d = len(shape)
    s = {}
    if kind in ("force", "grad"):
        chi, _ = _body(case, g)
        s["chi"] = chi.to(torch.uint8)
        amp = 0.2 if case.get("model") == "nonlinear" else 1e-3
        s["u"] = _waves(shape, d, g, amp).to(dt)
        if kind == "grad":
            s["s"] = (1.0 + _waves(shape, 1, g, 0.3)[0]).to(dt)
            s["gL"] = _waves(shape, d, g, 1.0, short=6.0).to(dt)
    elif kind == "dynamics":
        chi, _ = _body(case, g, hole=False)
        s["chi"] = chi.to(torch.uint8)
        lam, tip, mid = _notch(case, chi)
        s["lam"] = lam.to(torch.uint8)
        # the opening field of a crack with its tip at the notch's (plane stress, nu = 1/3, E = 1), scaled to
        # ``load`` times the critical stretch at a horizon from the tip and fading out over 8 horizons, on top of
        # smooth waves that run through the plate
        x1, x2 = _axis(shape, 0) - tip, _axis(shape, 1) - mid
        r, th = torch.sqrt(x1 * x1 + x2 * x2), torch.atan2(x2, x1)
        k = 0.5 * case["load"] * 1e-3 * math.sqrt(case["delta"]) / 0.75
        k = k * torch.sqrt(r) * torch.exp(-0.5 * (r / (8 * case["delta"])) ** 2)
        u1 = k * torch.cos(th / 2) * (1.0 + 2 * torch.sin(th / 2) ** 2)
        u2 = k * torch.sin(th / 2) * (3.0 - 2 * torch.cos(th / 2) ** 2)
        s["u"] = ((torch.stack([u1, u2]) + _waves(shape, 2, g, 2e-4, long=200.0, short=60.0)) * chi).to(dt)
        s["v"] = (_waves(shape, 2, g, 4e-4, long=200.0, short=60.0) * chi).to(dt)
        n2, m = shape[0], int(case["delta"])
        i2 = _axis(shape, 1)
        b = torch.zeros((2,) + shape, dtype=torch.float64, device=DEV)
        pull = 2e-5 * case["load"] * g.uniform(0.5, 1.0) / case["delta"]
        b[1] = (((i2 >= n2 - 2 * m) & chi).double() - ((i2 < 2 * m) & chi).double()) * pull
        s["b"] = b.to(dt)
    elif kind == "static":
        chi, ext = _body(case, g)
        om, b = _clamped(chi, ext, case, g)
        s["chi"], s["om"], s["b"] = chi.to(torch.uint8), torch.stack([om] * d).to(torch.uint8), b
    elif kind == "relax":
        s["items"] = []
        for k in range(case["count"]):
            pad = int(case["n"].split("x")[0]) >> (1 if k % 3 == 0 else 0)
            side = int(g.integers(pad // 2 + 8, pad + 1))
            one = dict(case, n="%dx%d" % (pad, pad), delta=float(g.integers(3, int(case["delta"]) + 1)),
                       fill=side / pad)
            chi, ext = _body(one, g)
            om, b = _clamped(chi, ext, one, g)
            s["items"].append((one, chi.to(torch.uint8), torch.stack([om] * d).to(torch.uint8), b))
    else:
        chi, _ = _body(case, g)
        s["chi"] = chi.to(torch.uint8)
        s["c"] = (1.0 + _waves(shape, 1, g, 0.2)[0]).to(dt)
        s["target"] = (_waves(shape, d, g, 1e-3) * chi).to(dt)
        c = [g.uniform(0.3, 0.6) * n for n in shape[::-1]]
        r2 = sum((_axis(shape, a) - c[a]) ** 2 for a in range(d))
        t = g.normal(size=d)
        pulse = torch.exp(-r2 / (2.0 * (2 * case["delta"]) ** 2)) * chi
        s["impulse"] = torch.stack([pulse * float(1e-2 * v) for v in t]).to(dt)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["kind"], s["case"] = case["kind"], case
    kind = case["kind"]
    if kind in ("force", "grad"):
        s["plan"] = pd.Plan(_problem(case, nu=0.4 if case.get("model") == "state" else 0.25), s["chi"])
        if kind == "grad":
            s["u"].requires_grad_(True)
            s["s"].requires_grad_(True)
    elif kind == "dynamics":
        s["plan"] = pd.Plan(_problem(case, rho=1.0, s0=1e-3, nu=1.0 / 3.0), s["chi"])
        s["plan"].set_energy_mode(not case.get("fp64"))  # single precision: the local sum, as its users need
        s["dt"] = _step(case)
        s["u0"], s["v0"], s["lam0"] = s["u"].clone(), s["v"].clone(), s["lam"].clone()
    elif kind == "static":
        s["plan"] = pd.Plan(_problem(dict(case, model="state"), E=1.0, nu=0.25), s["chi"], s["om"])
        s["u"] = torch.zeros_like(s["b"])
    elif kind == "relax":
        s["batch"] = pd.Batch([_problem(one) for one, _, _, _ in s["items"]], [chi for _, chi, _, _ in s["items"]],
                              [om for _, _, om, _ in s["items"]])
        s["b"] = [b for _, _, _, b in s["items"]]
        s["u"] = [torch.zeros_like(b) for b in s["b"]]
    else:
        s["plan"] = pd.Plan(_problem(case, rho=1.0), s["chi"])
        s["dt"] = _step(case)
        s["c"].requires_grad_(True)
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "force":
        return s["plan"].force(s["u"], want_energy=bool(case.get("energy")))
    if kind == "grad":
        L = autograd.pd_force(s["plan"], s["u"], s["s"])
        gu, gs = torch.autograd.grad(L, (s["u"], s["s"]), s["gL"])
        return L.detach(), gu, gs
    if kind == "dynamics":
        # a run restarts from its saved state
        s["u"].copy_(s["u0"])
        s["v"].copy_(s["v0"])
        s["lam"].copy_(s["lam0"])
        s["plan"].step_verlet(s["u"], s["v"], s["lam"], s["b"], None, dt=s["dt"], nsteps=case["steps"])
        return s["u"], s["v"], s["lam"]
    if kind == "static":
        s["u"].zero_()
        s["plan"].solve_static(s["u"], s["b"], None, rtol=case["rtol"], max_iter=50000)
        return s["u"]
    if kind == "relax":
        for u in s["u"]:
            u.zero_()
        s["batch"].solve_dr(s["u"], s["b"], None, rtol=case["rtol"], max_iter=400000)
        return list(s["u"])
    loss = autograd.verlet_loss(s["plan"], s["c"], s["target"], s["impulse"], s["dt"], case["steps"],
                                checkpoint_every=4)
    g, = torch.autograd.grad(loss, s["c"])
    return loss.detach(), g


# ---------------------------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------------------------

def _force_work(shape, item, fields_in, fields_out, flops_fields):
    """Bytes: each node field read or written once and the body mask; flops: 2.5 N log2 N a real transform."""
    n = float(np.prod(shape))
    return n * (item * (fields_in + fields_out) + 1), 2.5 * n * math.log2(n) * flops_fields


def work(case):
    shape = _shape(case)
    d, item = len(shape), 8 if case.get("fp64") else 4
    kind, model = case["kind"], case.get("model", "bond")
    nsym = d * (d + 1) // 2
    if kind == "force":
        e = bool(case.get("energy"))
        tr = 2 * d + (nsym + 1 if e else 0)
        if model == "state":
            tr = 2 * d + 2
        if model == "nonlinear":
            tr = (2 * d + nsym) + (2 * d + d * d + nsym)
        by, fl = _force_work(shape, item, d, d + (1 if e else 0), tr)
    elif kind == "grad":
        # forward: u, s -> L; backward: u, s, gL -> gu, gs
        b1, f1 = _force_work(shape, item, d + 1, d, 2 * d)
        b2, f2 = _force_work(shape, item, 2 * d + 1, d + 1, (2 * d + nsym) + (2 * d + 1))
        by, fl = b1 + b2, f1 + f2
    elif kind == "dynamics":
        # a step reads and writes u, v, reads b and lambda; it transforms v u_j forth and back
        by, fl = _force_work(shape, item, 3 * d, 2 * d, 2 * d + (nsym + 1 if case.get("fp64") else 0))
        by, fl = by * case["steps"], fl * case["steps"]
    elif kind in ("static", "relax"):
        # conjugate gradients take about 10 iterations per node layer of the longest side here, relaxation some 60
        # steps; an iteration reads and writes three vectors of FP32 and applies the operator
        if kind == "static":
            by, fl = _force_work(shape, 4, 4 * d, 3 * d, 2 * d)
            k = 10 * max(shape)
        else:
            by, fl = _force_work(shape, 4, 4 * d, 3 * d, 2 * d)
            by, fl, k = by * 0.6 * case["count"], fl * 0.6 * case["count"], 60 * max(shape)
        by, fl = by * k, fl * k
    else:
        # forward, the recomputed segment, and the reverse sweep's adjoint, per step
        b1, f1 = _force_work(shape, item, 2 * d + 1, 2 * d, 2 * d)
        b2, f2 = _force_work(shape, item, 3 * d + 1, d + 1, (2 * d + nsym) + (2 * d + 1))
        by, fl = (2 * b1 + b2) * case["steps"], (2 * f1 + f2) * case["steps"]
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------------------------------------------
# The same results in 64 bits, by torch's own transforms
# ---------------------------------------------------------------------------------------------------------------

def _bonds(d, delta):
    """Integer offsets within the horizon (spacing 1)."""
    r = int(math.floor(delta + 1e-9))
    ax = np.arange(-r, r + 1)
    o = np.stack([v.ravel() for v in np.meshgrid(*([ax] * d), indexing="ij")], 1)
    q = (o * o).sum(1)
    return o[(q > 0) & (q <= delta * delta * (1 + 1e-12))].astype(np.float64)


def _alpha(case, d):
    delta = case["delta"]
    if case.get("model") == "state" or case["kind"] == "static":
        nu = 0.4 if case.get("model") == "state" else 0.25
        r = np.sqrt((_bonds(d, delta) ** 2).sum(1))
        return 30.0 / (2 * (1 + nu)) / float(r.sum())
    return 9.0 / (math.pi * delta ** 3) if d == 2 else 12.0 / (math.pi * delta ** 4)


def _step(case):
    """0.8 of a bound of the stable time step: the symbol is at most twice the kernel's sum, isotropic here."""
    d = len(_shape(case))
    r = np.sqrt((_bonds(d, case["delta"]) ** 2).sum(1))
    trace = float((_alpha(case, d) / r).sum())
    return 0.8 * 2.0 / math.sqrt(2.0 * trace / d)


class _Exact:
    """Horizon sums as FP64 FFT products on the periodic box: corr(K)(f)(x) = sum_xi K(xi) f(x + xi)."""

    def __init__(self, shape, delta, alpha):
        self.shape, self.d = shape, len(shape)
        self.dims = tuple(range(-self.d, 0))
        self.o = _bonds(self.d, delta)
        self.r = np.sqrt((self.o ** 2).sum(1))
        self.alpha = alpha
        # grid axis of x_(a+1) is -(a + 1)
        self.at = tuple(torch.tensor(self.o[:, self.d - 1 - k].astype(np.int64) % shape[k], device=DEV)
                        for k in range(self.d))
        self.hat = {}

    def kernel(self, key, values):
        if key not in self.hat:
            k = torch.zeros(self.shape, dtype=torch.float64, device=DEV)
            k[self.at] = torch.tensor(values, device=DEV)
            self.hat[key] = torch.conj(torch.fft.rfftn(k)).resolve_conj()
        return self.hat[key]

    def C(self, i, j):
        i, j = min(i, j), max(i, j)
        h = self.kernel(("C", i, j), self.alpha * self.o[:, i] * self.o[:, j] / self.r ** 3)
        return h.real  # the kernel is even

    def f(self, x):
        return torch.fft.rfftn(x, dim=self.dims)

    def b(self, x):
        return torch.fft.irfftn(x, s=self.shape, dim=self.dims)

    def G(self, v):
        """sum_xi C_ij(xi) v(x + xi), all components."""
        vh = self.f(v)
        return {(i, j): self.b(self.C(i, j) * vh) for i in range(self.d) for j in range(i, self.d)}

    def force(self, u, v, G=None, energy=False):
        """L_i = v sum C_ij v' (u'_j - u_j); W = 1/2 v sum v' eta.C.eta."""
        d = self.d
        G = G or self.G(v)
        g = lambda i, j: G[min(i, j), max(i, j)]  # noqa: E731
        uh = [self.f(v * u[j]) for j in range(d)]
        y = [self.b(sum(self.C(i, j) * uh[j] for j in range(d))) for i in range(d)]
        Gu = [sum(g(i, j) * u[j] for j in range(d)) for i in range(d)]
        L = torch.stack([v * (y[i] - Gu[i]) for i in range(d)])
        if not energy:
            return L
        t = sum((1 if i == j else 2) * self.C(i, j) * self.f(v * u[i] * u[j])
                for i in range(d) for j in range(i, d))
        W = 0.5 * v * (self.b(t) + sum(u[i] * (Gu[i] - 2 * y[i]) for i in range(d)))
        return L, W


def _exact_force(case, s):
    shape = _shape(case)
    d = len(shape)
    chi, u = s["chi"].double(), s["u"].double()
    e = _Exact(shape, case["delta"], _alpha(case, d))
    model = case.get("model", "bond")
    if model == "bond":
        return e.force(u, chi, energy=bool(case.get("energy")))
    if model == "state":
        kappa, mu, m0 = 1.0 / (3 * 0.2), 1.0 / 2.8, float(e.r.sum())
        L = e.force(u, chi)
        gk = lambda i: e.kernel(("g", i), e.o[:, i] / e.r)  # noqa: E731  g = omega xi
        ch = e.f(chi)
        q = [e.b(gk(i) * ch) for i in range(3)]
        m = chi * e.b(e.kernel("m", e.r) * ch)
        th = sum(e.b(gk(i) * e.f(chi * u[i])) - q[i] * u[i] for i in range(3))
        th = torch.where(chi > 0, 3 * chi * th / torch.where(chi > 0, m, 1.0), 0.0)
        tv = e.f(th)
        ka = (3 * kappa - 5 * mu) / m0
        return L + torch.stack([chi * ka * (th * q[i] + e.b(gk(i) * tv)) for i in range(3)])
    # nonlinear bond: f = c/2 (|xi + eta|^2 - |xi|^2) (xi + eta), c = alpha / |xi|^3, summed bond by bond
    L = torch.zeros_like(u)
    for o, r in zip(e.o, e.r):
        sh = tuple(int(-v) for v in o)
        roll = lambda x: torch.roll(x, sh, dims=tuple(-1 - a for a in range(d)))  # noqa: E731
        w = e.alpha / r ** 3 * chi * roll(chi)
        eta = [roll(u[j]) - u[j] for j in range(d)]
        st = sum(o[j] * eta[j] + 0.5 * eta[j] ** 2 for j in range(d))
        for j in range(d):
            L[j] += w * st * (o[j] + eta[j])
    return L


def _exact_cg(shape, delta, alpha, chi, om, b):
    """Conjugate gradients in 64 bits on -chi_Omega L(chi_Omega e) = chi_Omega b, restarted on the true residual."""
    e = _Exact(shape, delta, alpha)
    chi, om = chi.double(), om.double()
    G = e.G(chi)
    A = lambda x: -om * e.force(x, chi, G)  # noqa: E731
    u = torch.zeros_like(b)
    rhs = om * b
    for _ in range(4):
        r = rhs - A(u)
        p, rr = r.clone(), float((r * r).sum())
        if rr <= 1e-28 * float((rhs * rhs).sum()):
            break
        stop = max(1e-16 * rr, 1e-28 * float((rhs * rhs).sum()))
        for it in range(20000):
            q = A(p)
            a = rr / (p * q).sum()
            u += a * p
            r -= a * q
            new = (r * r).sum()
            p = r + (new / rr) * p
            rr = new
            if it % 32 == 31 and float(rr) <= stop:
                break
        rr = float(rr)
    return u


def exact(case, seed):
    s = _inputs(case, seed)
    shape, kind = _shape(case), case["kind"]
    d = len(shape)
    if kind == "force":
        return _exact_force(case, s)
    if kind == "grad":
        e = _Exact(shape, case["delta"], _alpha(case, d))
        chi = s["chi"].double()
        u, w = s["u"].double().requires_grad_(True), s["s"].double().requires_grad_(True)
        L = e.force(u, chi * w)
        gu, gs = torch.autograd.grad(L, (u, w), s["gL"].double())
        return L.detach(), gu, gs
    if kind == "dynamics":
        e = _Exact(shape, case["delta"], _alpha(case, d))
        chi, u, v, b = s["chi"].double(), s["u"].double(), s["v"].double(), s["b"].double()
        lam, h, dt = s["lam"].double(), 0.5 * _step(case), _step(case)
        wc = 0.5 * e.alpha * 1e-6 * float(e.r.sum())
        L, W = e.force(u, chi * lam, energy=True)
        for _ in range(case["steps"]):
            v = v + h * (L + b)
            u = chi * (u + dt * v)
            lam = lam * torch.where((chi > 0) & (W > wc), 0.0, 1.0)
            L, W = e.force(u, chi * lam, energy=True)
            v = chi * (v + h * (L + b))
        return u, v, None
    if kind == "static":
        return _exact_cg(shape, case["delta"], _alpha(case, d), s["chi"], s["om"], s["b"])
    if kind == "relax":
        return [_exact_cg(_shape(one), one["delta"], _alpha(one, 2), chi, om, b) for one, chi, om, b in s["items"]]
    e = _Exact(shape, case["delta"], _alpha(case, d))
    chi, c = s["chi"].double(), s["c"].double().requires_grad_(True)
    w, h, dt = chi * torch.sqrt(c), 0.5 * _step(case), _step(case)
    G = e.G(w)
    u, v, f = torch.zeros_like(s["target"]).double(), torch.zeros_like(s["target"]).double(), s["impulse"].double()
    L = torch.zeros_like(u)
    for _ in range(case["steps"]):
        v = v + h * (L + f)
        u = chi * (u + dt * v)
        f = torch.zeros_like(f)
        L = e.force(u, w, G)
        v = chi * (v + h * L)
    loss = ((u - s["target"].double()) ** 2).sum()
    g, = torch.autograd.grad(loss, c)
    return loss.detach(), g
