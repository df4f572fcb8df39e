"""Measured cases: the work a program has this package do, through its public
entry points.

Every case is one call chain of `paper_1410_1764_gb300.api` on FP64 data: RK4
steps of the scalar wave (two-variable and first-order forms, several
finite-difference orders), of the variable-speed wave and of the BSSN system
on one periodic grid; single right-hand sides; batched patches; two-level mesh
refinement; constraints; and the discrete adjoint (forward and reverse).  Grid
sizes run from a few thousand points, where latency and launches count, to
the largest configured grids, with ragged sizes between them.

`exact` evaluates the same discretisation with double-double arithmetic
(pairs of 64-bit floats) in plain torch, so its own rounding is negligible
against that of a 64-bit evaluation.
"""
import math
from fractions import Fraction

import torch

from paper_1410_1764_gb300 import api

DEV = "cuda"
FLAT = (0, 1, 0, 0, 1, 0, 1, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 1, 0, 0, 0, 0, 0, 0)
NV = {"wave": 2, "wave1": 5, "varc": 2, "adjoint": 2}
EPS, ETA = 0.1, 2.0  # dissipation and Gamma-driver damping: the package's defaults


def listed():
    return [
        # the small scalar-wave run: 100 steps of a 32^3 plane wave, a step's latency counts
        dict(name="wave_32", kind="wave", order=4, nx=32, ny=32, nz=32, steps=100),
        # an odd-sized scalar wave of a quarter million points (a block of a multi-block driver)
        dict(name="wave_ragged", kind="wave", order=4, nx=61, ny=75, nz=53, steps=20),
        # the large scalar-wave run: Gaussian pulses on 256^3
        dict(name="wave_256", kind="wave", order=4, nx=256, ny=256, nz=256, steps=10),
        # high-order differencing, two-variable form
        dict(name="wave_o8", kind="wave", order=8, nx=128, ny=128, nz=128, steps=10),
        # first-order form of the wave equation, order 6, odd sizes
        dict(name="wave1_o6", kind="wave1", order=6, nx=117, ny=90, nz=131, steps=10),
        # forward propagation through a variable medium
        dict(name="varc_forward", kind="varc", order=4, nx=128, ny=128, nz=128, steps=20),
        # gradient of a receiver misfit: forward with checkpoints, then the reverse sweep
        dict(name="adjoint", kind="adjoint", order=4, nx=128, ny=128, nz=128, steps=50, ckpt=10, nrecv=512),
        # one right-hand side of a small odd-sized Einstein grid, as a caller with its own integrator asks for it
        dict(name="bssn_rhs_small", kind="bssn_rhs", nx=37, ny=29, nz=23, tuned=False),
        # the headline workload: RK4 steps of the Einstein equations, tuned and specialised
        dict(name="bssn_128", kind="bssn", nx=128, ny=128, nz=128, steps=2, tuned=True),
        # many small uneven grids advanced together (a multi-block driver)
        dict(name="bssn_patches", kind="patches", npatch=16, lo=16, hi=96, dims_seed=3, steps=2),
        # two refinement levels with subcycling, eight boxes
        dict(name="bssn_amr", kind="amr", nc=96, lo=8, hi=20, boxes_seed=5, steps=1),
        # analysis: constraints of an evolved state
        dict(name="bssn_constraints", kind="constraints", nx=128, ny=128, nz=128),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, lo, hi):
    n = [_logint(rng, lo, hi) for _ in range(3)]
    if rng.random() < 0.35:  # cubes and power-of-two sides are common
        n = [n[0]] * 3
    if rng.random() < 0.25:
        n = [max(32, 32 * (v // 32)) for v in n]
    return dict(nx=n[0], ny=n[1], nz=n[2])


def draw(rng):
    kind = rng.choice(["wave", "wave", "wave1", "varc", "adjoint", "bssn_rhs", "bssn", "patches", "amr",
                       "constraints"])
    if kind in ("wave", "wave1"):
        d = _dims(rng, 16, 224)
        return dict(kind=kind, order=rng.choice([2, 4, 4, 6, 8]), steps=rng.randint(2, 12), **d)
    if kind == "varc":
        return dict(kind=kind, order=4, steps=rng.randint(2, 20), **_dims(rng, 16, 160))
    if kind == "adjoint":
        return dict(kind=kind, order=4, steps=rng.randint(3, 24), ckpt=rng.randint(1, 8),
                    nrecv=rng.randint(1, 600), **_dims(rng, 16, 112))
    if kind == "bssn_rhs":
        return dict(kind=kind, tuned=rng.random() < 0.5, **_dims(rng, 12, 112))
    if kind == "bssn":
        return dict(kind=kind, steps=rng.randint(1, 2), tuned=rng.random() < 0.7, **_dims(rng, 12, 112))
    if kind == "patches":
        return dict(kind=kind, npatch=rng.randint(2, 12), lo=rng.randint(8, 16), hi=rng.randint(24, 96),
                    dims_seed=rng.randint(0, 10 ** 6), steps=rng.randint(1, 2))
    if kind == "amr":
        lo = rng.randint(4, 8)
        return dict(kind=kind, nc=rng.randint(48, 96), lo=lo, hi=lo + rng.randint(0, 8),
                    boxes_seed=rng.randint(0, 10 ** 6), steps=1)
    return dict(kind=kind, **_dims(rng, 12, 128))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _axes(n):
    """Coordinates in [0, 1) broadcastable as (z, y, x)."""
    nx, ny, nz = n
    ar = lambda m: torch.arange(m, device=DEV, dtype=torch.float64) / m  # noqa: E731
    return ar(nx)[None, None, :], ar(ny)[None, :, None], ar(nz)[:, None, None]


def _pulses(n, g):
    """Eight Gaussian pulses of width 0.05 at random places."""
    X = _axes(n)
    c, a = _rand(g, 8, 3).tolist(), _randn(g, 8).tolist()
    u = torch.zeros(n[2], n[1], n[0], device=DEV, dtype=torch.float64)
    for ci, ai in zip(c, a):
        e = ai
        for q, cq in zip(X, ci):
            r = q - cq
            r = r - torch.round(r)
            e = e * torch.exp(-0.5 * (r / 0.05) ** 2)
        u = u + e
    return u


def _modes(n, g, count):
    """`count` smooth periodic fields: a few long waves each, max about 1."""
    x, y, z = _axes(n)
    out = torch.empty(count, n[2], n[1], n[0], device=DEV, dtype=torch.float64)
    for v in range(count):
        f = torch.zeros(n[2], n[1], n[0], device=DEV, dtype=torch.float64)
        ph, am = _rand(g, 3).tolist(), _randn(g, 3).tolist()
        k = torch.randint(-2, 3, (3, 3), generator=g, device=DEV).tolist()
        for (a, b, c), p, m in zip(k, ph, am):
            f += m / 3 * torch.sin(2 * math.pi * (a * x + b * y + c * z + p))
        out[v] = f
    return out


def _pad(a, g):
    """Interior data with periodic ghost layers."""
    for d in (-1, -2, -3):
        i = torch.arange(-g, a.shape[d] + g, device=a.device) % a.shape[d]
        a = a.index_select(a.dim() + d, i)
    return a.contiguous()


def _zpad(a, g):
    return torch.nn.functional.pad(a, (g,) * 6)


def _bssn_interior(n, g):
    """Flat space with smooth perturbations of amplitude 1e-2 and the
    configured 1e-10 noise on every variable."""
    flat = torch.tensor(FLAT, device=DEV, dtype=torch.float64)[:, None, None, None]
    noise = 2e-10 * (_rand(g, 24, n[2], n[1], n[0]) - 0.5)
    return flat + 1e-2 * _modes(n, g, 24) + noise


def _size(case):
    return case["nx"], case["ny"], case["nz"]


def _ghosts(case):
    return max(2, case["order"] // 2)


def _wave_interior(case, g):
    n = _size(case)
    if case["kind"] == "wave" and max(n) <= 32:  # the small run's plane wave
        x, y, z = _axes(n)
        ph = 2 * math.pi * (x + y + z + float(_rand(g, 1)))
        w = 2 * math.pi * math.sqrt(3.0)
        return torch.stack([torch.sin(ph), -w * torch.cos(ph)])
    st = torch.zeros(NV[case["kind"]], n[2], n[1], n[0], device=DEV, dtype=torch.float64)
    st[0] = _pulses(n, g)
    if case["kind"] == "wave1":  # moving pulses: every field is live
        st[1] = _pulses(n, g)
        st[2:] = _modes(n, g, 3)
    return st


def _patch_dims(case):
    g = torch.Generator()
    g.manual_seed(case["dims_seed"])
    return [tuple(v) for v in torch.randint(case["lo"], case["hi"] + 1, (case["npatch"], 3), generator=g).tolist()]


def _amr_boxes(case):
    """Eight boxes, one per octant of the coarse grid, of uneven sides."""
    g = torch.Generator()
    g.manual_seed(case["boxes_seed"])
    pick = lambda a, b: int(torch.randint(a, b + 1, (1,), generator=g))  # noqa: E731
    nc, half, boxes = case["nc"], case["nc"] // 2, []
    for o in range(8):
        lo, hi = [], []
        for d in range(3):
            s = pick(case["lo"], case["hi"])
            oc = (o >> d) & 1
            a = pick(max(5, oc * half), min((oc + 1) * half, nc - 6) - s)
            lo.append(a)
            hi.append(a + s)
        boxes.append((tuple(lo), tuple(hi)))
    return boxes


def _inputs(case, seed):
    """Interior data of the case, a dict of tensors."""
    g, kind = _gen(seed), case["kind"]
    if kind in ("wave", "wave1"):
        return dict(state=_wave_interior(case, g))
    if kind in ("varc", "adjoint"):
        n = _size(case)
        c = 1.0 + 0.2 * _modes(n, g, 1)[0].clamp(-1, 1)
        u0 = torch.stack([_pulses(n, g), torch.zeros(n[2], n[1], n[0], device=DEV, dtype=torch.float64)])
        out = dict(state=u0, c=c)
        if kind == "adjoint":  # receiver traces: places and observed values at the field's scale
            nr = min(case["nrecv"], n[0] * n[1] * n[2])
            out["recv"] = torch.randperm(n[0] * n[1] * n[2], generator=g, device=DEV)[:nr].cpu()
            out["data"] = 0.3 * _randn(g, nr).cpu()
        return out
    if kind in ("bssn", "bssn_rhs", "constraints"):
        return dict(state=_bssn_interior(_size(case), g))
    if kind == "patches":
        return dict(states=[_bssn_interior(n, g) for n in _patch_dims(case)])
    nc, fine = case["nc"], []  # amr: both levels sample the same smooth fields
    flat = torch.tensor(FLAT, device=DEV, dtype=torch.float64)[:, None, None, None]
    whole = flat + 1e-2 * _modes((2 * nc,) * 3, g, 24)
    coarse = whole[:, ::2, ::2, ::2].contiguous()
    for lo, hi in _amr_boxes(case):
        fine.append(whole[:, 2 * lo[2]:2 * hi[2], 2 * lo[1]:2 * hi[1], 2 * lo[0]:2 * hi[0]].contiguous())
    return dict(coarse=coarse, fine=fine)


def _dx(case):
    if case["kind"] == "patches":
        return 1.0 / 64
    return 1.0 / case["nc"] if case["kind"] == "amr" else 1.0 / case["nx"]


def _dt(case):
    return 0.25 * _dx(case)


def prepare(case, seed):
    kind, x, h = case["kind"], _inputs(case, seed), _dx(case)
    st = dict(case=case, dt=_dt(case))
    if kind in ("wave", "wave1"):
        g = _ghosts(case)
        sysm = api.make_system(api.WAVE if kind == "wave" else api.WAVE1, *_size(case), h,
                               params=api.default_params(fd_order=case["order"]), nghost=g)
        st.update(sys=sysm, y=_pad(x["state"], g))
        sysm.autotune(st["y"])
    elif kind == "varc":
        sysm = api.make_system(api.WAVE_VARC, *_size(case), h)
        sysm.set_speed(_pad(x["c"], 2))
        st.update(sys=sysm, y=_pad(x["state"], 2))
        sysm.autotune(st["y"])
    elif kind == "adjoint":
        n = _size(case)
        r = x["recv"]
        k, j, i = r // (n[0] * n[1]), (r // n[0]) % n[1], r % n[0]
        recv = ((k + 2) * (n[1] + 4) + j + 2) * (n[0] + 4) + i + 2
        st.update(sys=api.make_system(api.WAVE_VARC, *n, h), u0=_pad(x["state"], 2).requires_grad_(),
                  c=_pad(x["c"], 2).requires_grad_(), recv=recv.numpy(), data=x["data"].numpy())
    elif kind in ("bssn", "bssn_rhs", "constraints"):
        sysm = api.make_system(api.BSSN, *_size(case), h)
        st.update(sys=sysm, y0=_pad(x["state"], 3))
        if case.get("tuned"):
            sysm.autotune(st["y0"])
            sysm.specialize()
        if kind == "bssn":
            st["y"] = st["y0"].clone()
    elif kind == "patches":
        b = api.Batch(_patch_dims(case), 3, h)
        st.update(batch=b, y0=[_pad(a, 3) for a in x["states"]], views=[b.state(p) for p in range(case["npatch"])])
    else:
        amr = api.AmrBoxes(api.BSSN, (case["nc"],) * 3, _amr_boxes(case), h)
        nb = len(amr.boxes)
        st.update(amr=amr, y0=[_pad(x["coarse"], 3)] + [_zpad(a, 12) for a in x["fine"]],
                  views=[amr.state(q) for q in range(nb + 1)])
        st["views"][0].copy_(st["y0"][0])
        amr.autotune()
    return st


def run(state):
    """One pass.  The wave systems advance in place from pass to pass, as a
    simulation does; the Einstein grids start each pass from the given state
    (an ensemble member), so that every pass sees data of the same kind."""
    case = state["case"]
    kind = case["kind"]
    if kind in ("wave", "wave1", "varc"):
        return state["sys"].rk4_step(state["y"], state["dt"], case["steps"])
    if kind == "adjoint":
        loss = api.WaveAdjoint.apply(state["u0"], state["c"], state["sys"], state["recv"], state["data"],
                                     state["dt"], case["steps"], case["ckpt"])
        gu, gc = torch.autograd.grad(loss, (state["u0"], state["c"]))
        return dict(loss=loss.detach(), grad_u0=gu, grad_c=gc)
    if kind == "bssn_rhs":
        return state["sys"].rhs(state["y0"])
    if kind == "constraints":
        return state["sys"].constraints(state["y0"])
    if kind == "bssn":
        state["y"].copy_(state["y0"])
        return state["sys"].rk4_step(state["y"], state["dt"], case["steps"])
    for v, y in zip(state["views"], state["y0"]):
        v.copy_(y)
    state["batch" if kind == "patches" else "amr"].step(state["dt"], case["steps"])
    return list(state["views"])


# ---------------------------------------------------------------------------
# work and tolerances
# ---------------------------------------------------------------------------
RHS_FLOPS = {"wave": {2: 21, 4: 27, 6: 45, 8: 57}, "wave1": {2: 19, 4: 31, 6: 43, 8: 55}}
BSSN_FLOPS, CONSTRAINT_FLOPS = 3760, 2695  # per point of one evaluation


def work(case):
    kind = case["kind"]
    if kind in ("wave", "wave1", "varc", "adjoint", "bssn", "bssn_rhs", "constraints"):
        pts = case["nx"] * case["ny"] * case["nz"]
    if kind in ("wave", "wave1"):
        nv = NV[kind]
        return dict(bytes=16 * nv * pts, flops=pts * case["steps"] * 4 * (RHS_FLOPS[kind][case["order"]] + 3.25 * nv))
    if kind == "varc":
        return dict(bytes=(16 * 2 + 8) * pts, flops=pts * case["steps"] * 4 * (49 + 6.5))
    if kind == "adjoint":  # forward, and the transpose of every stage
        return dict(bytes=8 * (2 + 1 + 2 + 1) * pts, flops=pts * case["steps"] * 4 * (49 + 6.5 + 110))
    if kind == "bssn_rhs":
        return dict(bytes=8 * 48 * pts, flops=BSSN_FLOPS * pts)
    if kind == "constraints":
        return dict(bytes=8 * 31 * pts, flops=CONSTRAINT_FLOPS * pts)
    if kind == "bssn":
        return dict(bytes=16 * 24 * pts, flops=pts * case["steps"] * 4 * (BSSN_FLOPS + 78))
    if kind == "patches":
        pts = sum(a * b * c for a, b, c in _patch_dims(case))
        return dict(bytes=16 * 24 * pts, flops=pts * case["steps"] * 4 * (BSSN_FLOPS + 78))
    pc = case["nc"] ** 3
    pf = sum(8 * math.prod(h - l for l, h in zip(lo, hi)) for lo, hi in _amr_boxes(case))
    return dict(bytes=16 * 24 * (pc + pf), flops=case["steps"] * (pc * 5 + pf * 8) * (BSSN_FLOPS + 78))


def tolerance(case):
    kind = case["kind"]
    # the rounding of a state at every stage, carried on with weights of order
    # one over the spacing; about four times the distance of the present
    # 64-bit evaluation from `exact` over the listed cases and some draws
    if kind == "wave1":
        return {"rel": 1e-15}
    if kind == "varc":
        return {"rel": 1e-14}
    if kind == "adjoint":
        return {"rel": 1e-13}
    if kind in ("bssn_rhs", "constraints"):
        return {"rel": 2e-15}
    return {"rel": 4e-14}


# ---------------------------------------------------------------------------
# the same discretisation in double-double arithmetic
# ---------------------------------------------------------------------------
class DD:
    """An unevaluated sum hi + lo of two float64 tensors (or of two floats)."""

    def __init__(self, hi, lo=None):
        self.hi = hi
        self.lo = torch.zeros_like(hi) if lo is None else lo

    @staticmethod
    def const(q):
        q = Fraction(q)
        hi = float(q)
        return DD(hi, float(q - Fraction(hi)))

    @staticmethod
    def _of(b):
        return b if isinstance(b, DD) else DD.const(b)

    @staticmethod
    def _fast(a, b):
        s = a + b
        return DD(s, b - (s - a))

    def __add__(self, b):
        b = DD._of(b)
        s = self.hi + b.hi
        t = s - self.hi
        e = (self.hi - (s - t)) + (b.hi - t)
        return DD._fast(s, e + (self.lo + b.lo))

    def __neg__(self):
        return DD(-self.hi, -self.lo)

    def __sub__(self, b):
        return self + (-DD._of(b))

    def __rsub__(self, b):
        return (-self) + b

    @staticmethod
    def _split(a):
        c = 134217729.0 * a
        h = c - (c - a)
        return h, a - h

    def __mul__(self, b):
        if isinstance(b, int) and b & (b - 1) == 0 and b > 0:
            return DD(self.hi * b, self.lo * b)
        b = DD._of(b)
        p = self.hi * b.hi
        ah, al = DD._split(self.hi)
        bh, bl = DD._split(b.hi)
        e = ((ah * bh - p) + ah * bl + al * bh) + al * bl
        return DD._fast(p, e + (self.hi * b.lo + self.lo * b.hi))

    __radd__ = __add__
    __rmul__ = __mul__

    def recip(self):
        r = DD(1.0 / self.hi)
        for _ in range(2):
            r = r + r * (1 - self * r)
        return r

    def exp(self):
        # e^(hi + lo) by a Taylor series of the argument over 256
        x = self * DD.const(Fraction(1, 256))
        s = DD.const(Fraction(1, math.factorial(10)))
        for k in range(9, -1, -1):
            s = x * s + Fraction(1, math.factorial(k))
        for _ in range(8):
            s = s * s
        return s

    def roll(self, m, dim):
        return DD(torch.roll(self.hi, -m, dim), torch.roll(self.lo, -m, dim))

    def __getitem__(self, i):
        return DD(self.hi[i], self.lo[i])

    def value(self):
        return self.hi + self.lo


def _stack(a):
    return DD(torch.stack([q.hi for q in a]), torch.stack([q.lo for q in a]))


def _weights(order, h):
    """Central weights of D1 (odd pairs) and D2 (centre differences), exact."""
    m, h = order // 2, Fraction(h)
    a, b = [], []
    for k in range(1, m + 1):
        w = Fraction(2 * (-1) ** (k + 1) * math.factorial(m) ** 2, math.factorial(m - k) * math.factorial(m + k))
        a.append(w / (2 * k) / h)
        b.append(w / k ** 2 / h ** 2)
    return a, b


class Stencils:
    """Periodic central differences on (z, y, x) fields; axis 0 is x."""

    def __init__(self, order, h):
        self.a, self.b = _weights(order, h)
        self.h = Fraction(h)

    def d1(self, f, ax):
        return self._sum([(w, f.roll(k, -1 - ax) - f.roll(-k, -1 - ax)) for k, w in enumerate(self.a, 1)])

    def d2(self, f, ax):
        return self._sum([(w, (f.roll(k, -1 - ax) - f) + (f.roll(-k, -1 - ax) - f)) for k, w in enumerate(self.b, 1)])

    def lap(self, f):
        return self.d2(f, 0) + self.d2(f, 1) + self.d2(f, 2)

    def dd(self, f, a, b):
        return self.d2(f, a) if a == b else self.d1(self.d1(f, a), b)

    def ko(self, f):
        s = None
        for ax in range(3):
            for k, w in ((1, 15), (2, -6), (3, 1)):
                t = ((f.roll(k, -1 - ax) - f) + (f.roll(-k, -1 - ax) - f)) * w
                s = t if s is None else s + t
        return s * (Fraction(EPS) / (64 * self.h))

    @staticmethod
    def _sum(terms):
        s = None
        for w, f in terms:
            s = f * w if s is None else s + f * w
        return s


def _rk4(y, dt, rhs, steps):
    dt = Fraction(dt)
    for _ in range(steps):
        k1 = rhs(y)
        k2 = rhs(y + k1 * (dt / 2))
        k3 = rhs(y + k2 * (dt / 2))
        k4 = rhs(y + k3 * dt)
        y = y + (k1 + k2 * 2 + k3 * 2 + k4) * (dt / 6)
    return y


def _wave_rhs(S):
    return lambda y: _stack([y[1], S.lap(y[0])])


def _wave1_rhs(S):
    return lambda y: _stack([y[1], S.d1(y[2], 0) + S.d1(y[3], 1) + S.d1(y[4], 2)] + [S.d1(y[1], a) for a in range(3)])


def _varc_rhs(S, s, G):
    def rhs(y):
        r = s * S.lap(y[0])
        for a in range(3):
            r = r + G[a] * S.d1(y[0], a)
        return _stack([y[1], r])
    return rhs


def _dot(a, b):
    s = None
    for x, y in zip(a, b):
        s = x * y if s is None else s + x * y
    return s


SYM = ((0, 1, 2), (1, 3, 4), (2, 4, 5))
R3 = range(3)


def _geometry(S, y):
    """Derivatives, inverse metric, Christoffels, Ricci tensor and curvature
    contractions of the conformal BSSN variables."""
    def sym(base):
        return [[y[base + SYM[i][j]] for j in R3] for i in R3]

    def grad(f):
        return [S.d1(f, a) for a in R3]

    def sym_of(fn):
        q = [[None] * 3 for _ in R3]
        for i in R3:
            for j in range(i, 3):
                q[i][j] = q[j][i] = fn(i, j)
        return q

    phi, gt, At, Xt = y[0], sym(1), sym(8), [y[14 + i] for i in R3]
    dphi, dK, dX = grad(phi), grad(y[7]), [grad(x) for x in Xt]
    dg = sym_of(lambda i, j: grad(gt[i][j]))
    co = sym_of(lambda i, j: gt[(i + 1) % 3][(j + 1) % 3] * gt[(i + 2) % 3][(j + 2) % 3]
                - gt[(i + 1) % 3][(j + 2) % 3] * gt[(i + 2) % 3][(j + 1) % 3])
    idet = _dot(gt[0], co[0]).recip()
    gu = sym_of(lambda i, j: co[i][j] * idet)
    half = Fraction(1, 2)
    Gl = [sym_of(lambda i, j, k=k: (dg[j][k][i] + dg[i][k][j] - dg[i][j][k]) * half) for k in R3]
    Gu = [sym_of(lambda i, j, k=k: _dot(gu[k], [Gl[l][i][j] for l in R3])) for k in R3]
    flat = [(a, b) for a in R3 for b in R3]
    tr = lambda A, B: _dot([A[a][b] for a, b in flat], [B[a][b] for a, b in flat])  # noqa: E731
    Gd = [tr(gu, Gu[k]) for k in R3]
    ddphi = sym_of(lambda i, j: S.dd(phi, i, j))
    Dphi = sym_of(lambda i, j: ddphi[i][j] - _dot([Gu[k][i][j] for k in R3], dphi))
    gphi = [_dot(gu[i], dphi) for i in R3]
    trD, phi2 = tr(gu, Dphi), _dot(gphi, dphi)
    C = [[[_dot(gu[l], Gl[j][k]) for l in R3] for k in R3] for j in R3]

    def ricci(i, j):
        r = tr(gu, [[S.dd(gt[i][j], a, b) for b in R3] for a in R3]) * (-half)
        for k in R3:
            r = r + (gt[k][i] * dX[k][j] + gt[k][j] * dX[k][i] + Gd[k] * (Gl[i][j][k] + Gl[j][i][k])) * half
            for l in R3:
                r = r + Gu[k][l][i] * C[j][k][l] + Gu[k][l][j] * C[i][k][l] + Gu[k][i][l] * C[k][j][l]
        return (r - Dphi[i][j] * 2 - gt[i][j] * trD * 2 + dphi[i] * dphi[j] * 4 - gt[i][j] * phi2 * 4)

    R = sym_of(ricci)
    Am = [[_dot(gu[i], [At[k][j] for k in R3]) for j in R3] for i in R3]
    Au = sym_of(lambda i, j: _dot(Am[i], gu[j]))
    return dict(locals())


def _bssn_rhs(S):
    third = Fraction(1, 3)

    def rhs(y):
        G = _geometry(S, y)
        gt, At, gu, Gu, Gd, Am, Au = (G[k] for k in ("gt", "At", "gu", "Gu", "Gd", "Am", "Au"))
        tr, grad, dphi, dK, gphi = (G[k] for k in ("tr", "grad", "dphi", "dK", "gphi"))
        K, al = y[7], y[17]
        be, B = [y[18 + i] for i in R3], [y[21 + i] for i in R3]
        dal, db = grad(al), [grad(b) for b in be]
        e4 = (y[0] * -4).exp()
        div = db[0][0] + db[1][1] + db[2][2]
        adv = lambda df: _dot(be, df)  # noqa: E731
        gal = _dot(gphi, dal)
        DDal = [[None] * 3 for _ in R3]
        ddal = [[None] * 3 for _ in R3]
        for i in R3:
            for j in range(i, 3):
                ddal[i][j] = ddal[j][i] = S.dd(al, i, j)
                DDal[i][j] = DDal[j][i] = (ddal[i][j] - _dot([Gu[k][i][j] for k in R3], dal)
                                           - (dphi[i] * dal[j] + dphi[j] * dal[i]) * 2 + gt[i][j] * gal * 2)
        out = [None] * 24
        out[0] = adv(dphi) + (div - al * K) * Fraction(1, 6)
        lap = e4 * (tr(gu, ddal) - _dot(Gd, dal) + gal * 2)
        out[7] = adv(dK) - lap + al * (tr(At, Au) + K * K * third)
        X = [[al * G["R"][i][j] - DDal[i][j] for j in R3] for i in R3]
        trX = tr(gu, X)
        for i in R3:
            for j in range(i, 3):
                s = SYM[i][j]
                bj, bi = [db[k][j] for k in R3], [db[k][i] for k in R3]
                out[1 + s] = (adv(G["dg"][i][j]) + _dot(gt[i], bj) + _dot(gt[j], bi) - gt[i][j] * div * (2 * third)
                              - al * At[i][j] * 2)
                out[8 + s] = (adv(grad(At[i][j])) + _dot(At[i], bj) + _dot(At[j], bi)
                              - At[i][j] * div * (2 * third) + e4 * (X[i][j] - gt[i][j] * trX * third)
                              + al * (K * At[i][j] - _dot(At[i], [Am[k][j] for k in R3]) * 2))
        ddiv = [None] * 3
        ddb = [[[None] * 3 for _ in R3] for _ in R3]
        for k in R3:
            for a in R3:
                for b in range(a, 3):
                    ddb[k][a][b] = ddb[k][b][a] = S.dd(be[k], a, b)
        for j in R3:
            ddiv[j] = ddb[0][0][j] + ddb[1][1][j] + ddb[2][2][j]
        for i in R3:
            ax = adv(G["dX"][i])
            r = (ax - _dot(Gd, db[i]) + Gd[i] * div * (2 * third) + tr(gu, ddb[i]) + _dot(gu[i], ddiv) * third
                 - _dot(Au[i], dal) * 2
                 + al * (tr(Gu[i], Au) + _dot(Au[i], dphi) * 6 - _dot(gu[i], dK) * (2 * third)) * 2)
            out[14 + i] = r
            out[18 + i] = adv(db[i]) + B[i] * Fraction(3, 4)
            out[21 + i] = adv(grad(B[i])) + (r - ax) - B[i] * Fraction(ETA)
        out[17] = adv(dal) - al * K * 2
        return _stack([out[v] + S.ko(y[v]) for v in range(24)])

    return rhs


def _constraints(S, y):
    G = _geometry(S, y)
    gu, Gu, Gd, Am, Au, At, tr = (G[k] for k in ("gu", "Gu", "Gd", "Am", "Au", "At", "tr"))
    e4, K = (y[0] * -4).exp(), y[7]
    out = [e4 * tr(gu, G["R"]) + K * K * Fraction(2, 3) - tr(At, Au)]
    dA = [[[None] * 3 for _ in R3] for _ in R3]
    for a in R3:
        for b in range(a, 3):
            dA[a][b] = dA[b][a] = G["grad"](At[a][b])
    for i in R3:
        m = tr(Gu[i], Au) + _dot(Au[i], G["dphi"]) * 6 - _dot(gu[i], G["dK"]) * Fraction(2, 3)
        for j in R3:
            # d_j of gu^ia gu^jb At_ab, with d gu = - gu dg gu
            m = m + _dot(gu[i], [_dot(gu[j], [dA[a][b][j] for b in R3]) for a in R3])
            m = m - _dot(gu[i], [_dot([Au[j][b] for b in R3], [G["dg"][a][b][j] for b in R3]) for a in R3])
            m = m - _dot(gu[j], [_dot([Au[i][a] for a in R3], [G["dg"][a][b][j] for a in R3]) for b in R3])
        out.append(m)
    return _stack(out + [G["Xt"][i] - Gd[i] for i in R3])


def _adjoint_exact(case, x):
    """Loss and gradients of the fully discrete map, reverse mode by hand."""
    S = Stencils(4, _dx(case))
    dt = Fraction(_dt(case))
    c = DD(x["c"])
    s = c * c
    G = [S.d1(s, a) for a in R3]
    rhs = _varc_rhs(S, s, G)
    y, states = DD(x["state"]), []
    for _ in range(case["steps"]):
        k1 = rhs(y)
        y2 = y + k1 * (dt / 2)
        k2 = rhs(y2)
        y3 = y + k2 * (dt / 2)
        k3 = rhs(y3)
        y4 = y + k3 * dt
        k4 = rhs(y4)
        states.append([q[0] for q in (y, y2, y3, y4)])
        y = y + (k1 + k2 * 2 + k3 * 2 + k4) * (dt / 6)
    r = x["recv"].to(DEV)
    u = DD(y[0].hi.flatten()[r], y[0].lo.flatten()[r]) - DD(x["data"].to(DEV))
    sq = u * u
    loss = sum((Fraction(a) + Fraction(b) for a, b in zip(sq.hi.tolist(), sq.lo.tolist())), Fraction(0)) / 2
    yb = DD(torch.zeros_like(x["state"]))
    yb.hi[0].view(-1)[r], yb.lo[0].view(-1)[r] = u.hi, u.lo
    sb = DD(torch.zeros_like(x["c"]))
    for n in range(case["steps"] - 1, -1, -1):
        nxt, total = None, yb
        for q, (wb, wn) in zip((3, 2, 1, 0), ((dt / 6, None), (dt / 3, dt), (dt / 3, dt / 2), (dt / 6, dt / 2))):
            kb = yb * wb if nxt is None else yb * wb + nxt * wn
            w, uq = kb[1], states[n][q]
            yu = S.lap(s * w)
            sb = sb + w * S.lap(uq)
            for a in R3:
                yu = yu - S.d1(G[a] * w, a)
                sb = sb - S.d1(w * S.d1(uq, a), a)
            nxt = _stack([yu, kb[0]])
            total = total + nxt
        yb = total
    gc = (c * sb) * 2
    return dict(loss=torch.tensor(float(loss), device=DEV, dtype=torch.float64), grad_u0=_zpad(yb.value(), 2),
                grad_c=_zpad(gc.value(), 2))


def exact(case, seed):
    kind = case["kind"]
    if kind == "amr":  # two levels with prolongation: no short plain form
        return None
    x, h = _inputs(case, seed), _dx(case)
    if kind == "adjoint":
        return _adjoint_exact(case, x)
    if kind in ("wave", "wave1", "varc"):
        S = Stencils(case["order"], h)
        if kind == "varc":
            c = DD(x["c"])
            s = c * c
            rhs = _varc_rhs(S, s, [S.d1(s, a) for a in R3])
        else:
            rhs = (_wave_rhs if kind == "wave" else _wave1_rhs)(S)
        return _pad(_rk4(DD(x["state"]), _dt(case), rhs, case["steps"]).value(), _ghosts(case))
    S = Stencils(4, h)
    if kind == "bssn_rhs":
        return _zpad(_bssn_rhs(S)(DD(x["state"])).value(), 3)
    if kind == "constraints":
        return _zpad(_constraints(S, DD(x["state"])).value(), 3)
    if kind == "bssn":
        return _pad(_rk4(DD(x["state"]), _dt(case), _bssn_rhs(S), case["steps"]).value(), 3)
    # patches are independent: two of them stand for all (some seconds each)
    return [_pad(_rk4(DD(a), _dt(case), _bssn_rhs(S), case["steps"]).value(), 3) if p < 2 else None
            for p, a in enumerate(x["states"])]
