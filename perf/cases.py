"""Performance cases of the propagators: modelling, adjoint modelling and FWI gradients as a
program calls them through ``paper_2004_10519_gb300``.

A case is a dict of plain values: the call (``op``), the propagator (``kind``), the physical grid,
the absorbing layer, the space order, the number of time steps and, for gradients, how the forward
wavefield is kept.  The time steps are fewer than a survey's thousands: every step costs the same,
so a few dozen of them time the call.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_2004_10519_gb300 as wp

KIND = {"tti": wp.PROP_TTI, "elastic": wp.PROP_ELASTIC, "acoustic": wp.PROP_ACOUSTIC,
        "elastic2d": wp.PROP_ELASTIC2D}
SNAP = {"full": wp.SNAP_FULL_FP32, "fp32": wp.SNAP_CKPT_FP32, "bf16": wp.SNAP_CKPT_BF16}
SPACING = {"tti": 12.5, "elastic": 10.0, "acoustic": 12.5, "elastic2d": 5.0}
VMIN, VMAX, EPS_MAX = 1.5, 4.5, 0.3        # km/s; Thomsen epsilon grows with vp


def _case(name, op, kind, nx, ny, nz, nbl, so, nt, snap="full", shots=1):
    c = {"op": op, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "nbl": nbl, "so": so, "nt": nt,
         "snap": snap, "shots": shots}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a near-surface or toy model, where launches and host work count
        _case("acoustic_forward_small", "forward", "acoustic", 60, 60, 60, 10, 8, 200),
        # the two-layer TTI workload of the repository (64^3 at space order 8, 150 steps)
        _case("tti_forward_small", "forward", "tti", 64, 64, 64, 10, 8, 150),
        # forward modelling of the elastic benchmark grid (256^3 + 20 cells, space order 8)
        _case("elastic_forward", "forward", "elastic", 256, 256, 256, 20, 8, 40),
        # adjoint modelling on a grid cut to a survey: odd sizes, rows of 139 points
        _case("elastic_adjoint_ragged", "adjoint", "elastic", 161, 131, 99, 20, 8, 60),
        # elastic FWI gradient (lambda, mu, b), one shot, full storage
        _case("elastic_gradient", "gradient", "elastic", 160, 160, 160, 20, 8, 40),
        # TTI forward modelling on the grid of the TTI gradient workload (400x400x300 + 40, so 12)
        _case("tti_forward", "forward", "tti", 400, 400, 300, 40, 12, 16),
        # TTI forward on odd sizes: a window cut out of a larger model, rows of 193 points
        _case("tti_forward_ragged", "forward", "tti", 201, 187, 113, 40, 12, 40),
        # TTI FWI gradient of one shot with FP32 checkpoints
        _case("tti_gradient", "gradient", "tti", 200, 200, 160, 40, 12, 40, "fp32"),
        # all five TTI parameters (m, eps, delta, theta, phi)
        _case("tti_gradient_aniso", "aniso", "tti", 96, 96, 80, 20, 8, 40),
        # one RTM shot: acoustic gradient on a window of the batched RTM workload
        _case("acoustic_gradient", "gradient", "acoustic", 320, 320, 300, 40, 12, 40, "fp32"),
        # the 2D marine workload (1701 x 701 + 40, space order 8)
        _case("elastic2d_forward", "forward", "elastic2d", 1701, 1, 701, 40, 8, 300),
        # many small TTI shots at once with 16-bit checkpoints (windows U[40, 80]^2 x 60 + 40)
        _case("tti_gradient_batch", "batch", "tti", 60, 60, 60, 40, 12, 40, "bf16", 8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op, kind = rng.choice([("forward", "acoustic"), ("forward", "tti"), ("forward", "elastic"),
                           ("adjoint", "elastic"), ("adjoint", "tti"), ("gradient", "elastic"),
                           ("gradient", "tti"), ("gradient", "acoustic"), ("aniso", "tti"),
                           ("forward", "elastic2d"), ("batch", "tti")])
    nbl = rng.choice([10, 20, 40])
    so = rng.choice([4, 8, 12])
    snap, shots = "full", 1
    if kind == "elastic2d":
        nx, ny, nz = _log_int(rng, 150, 2000), 1, _log_int(rng, 100, 800)
        cells = (nx + 2 * nbl) * (nz + 2 * nbl)
        nt = min(400, max(100, int(3e8 / cells)))
        return _case("", op, kind, nx, ny, nz, nbl, so, nt)
    if op == "batch":
        # one depth for every window, as in a survey; rows of a multiple of 4 points
        nbl, shots, snap = rng.choice([20, 40]), rng.choice([4, 8, 12]), "bf16"
        c = _case("", op, kind, _log_int(rng, 40, 70), _log_int(rng, 40, 70), 4 * rng.randint(12, 18), nbl,
                  rng.choice([8, 12]), 1, snap, shots)
        return dict(c, nt=min(rng.randint(24, 44), int(1.2e11 / work(c)["bytes"])))
    big = 280 if op in ("gradient", "aniso") else 360
    nx, ny, nz = _log_int(rng, 40, big), _log_int(rng, 40, big), _log_int(rng, 40, 260)
    if op == "aniso":
        nz += -nz % 2              # whole 16-byte rows, which every option of this call has
        nz += (nz + 2 * nbl) % 4
    if op == "gradient":
        snap = rng.choice(["full", "fp32"])
    cells = (nx + 2 * nbl) * (ny + 2 * nbl) * (nz + 2 * nbl)
    nt = min(150, max(16, int((3e8 if op in ("gradient", "aniso") else 6e8) / cells)))
    return _case("", op, kind, nx, ny, nz, nbl, so, nt, snap, shots)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _dt(case):
    v = 1000.0 * VMAX * (math.sqrt(1 + 2 * EPS_MAX) if case["kind"] == "tti" else 1.0)
    return float(np.float32(0.4 * SPACING[case["kind"]] / v))


def _noise(shape, gen):
    """Smooth noise in [0, 1]: white noise on every eighth point, interpolated."""
    coarse = torch.rand([1, 1] + [n // 8 + 2 for n in shape], generator=gen, device="cuda")
    return torch.nn.functional.interpolate(coarse, size=shape, mode="trilinear", align_corners=True)[0, 0]


def _model(case, gen):
    """Layered velocity growing with depth plus smooth noise, and what follows from it."""
    shape = (case["nx"], case["ny"], case["nz"])
    z = torch.arange(shape[2], device="cuda") / max(shape[2] - 1, 1)
    layer = VMIN + (VMAX - VMIN) * torch.clamp(torch.floor(10 * z), max=9.0) / 9
    vp = torch.clamp(layer + 1.5 * (_noise(shape, gen) - 0.5), VMIN, VMAX)
    if case["kind"] == "acoustic":
        return [vp]
    if case["kind"] == "tti":
        eps = EPS_MAX * (vp - VMIN) / (VMAX - VMIN)
        return [vp, eps, 0.5 * eps, math.radians(40) * _noise(shape, gen), math.radians(90) * _noise(shape, gen)]
    vs, rho = vp / 1.9, 0.31 * (1000.0 * vp) ** 0.25
    if case["kind"] == "elastic2d":          # marine: 30 m of water over the layers
        water = (torch.arange(shape[2], device="cuda") * SPACING["elastic2d"] < 30.0).expand(shape)
        vp, vs = torch.where(water, 1.5, vp), torch.where(water, 0.0, vs)
        rho = torch.where(water, 1.02, rho)
    return [a.float().contiguous() for a in (vp, vs, rho)]


def _shot(case, seed, nx, ny):
    """Source, wavelet, receivers and (gradients, adjoint) the traces of one shot."""
    rng = np.random.default_rng(seed)
    kind, h, nt, dt = case["kind"], SPACING[case["kind"]], case["nt"], _dt(case)
    nsrc = 16 if case["op"] == "adjoint" else 1
    src = np.zeros((nsrc, 3), np.float32)
    src[:, 0] = h * (nx / 2 + rng.uniform(-0.2 * nx, 0.2 * nx, nsrc))
    src[:, 1] = 0.0 if kind == "elastic2d" else h * (ny / 2 + rng.uniform(-0.2 * ny, 0.2 * ny, nsrc))
    src[:, 2] = 2 * h
    every = 2 if kind == "elastic2d" else 4
    x = h * every * np.arange((nx - 1) // every + 1)
    y = h * every * np.arange((ny - 1) // every + 1)
    rec = np.stack([a.ravel() for a in np.meshgrid(x, y, [h], indexing="ij")], 1).astype(np.float32)
    f0 = max(12.0, 2.0 / (nt * dt))          # the wavelet fits the record
    t = np.arange(nt) * dt
    pulse = lambda tau: (1 - 2 * (math.pi * f0 * tau) ** 2) * np.exp(-(math.pi * f0 * tau) ** 2)  # noqa: E731
    wav = (pulse(t - 1 / f0)[None] * rng.uniform(0.8, 1.2, (nsrc, 1))).astype(np.float32)
    # recorded traces: the direct arrival of a homogeneous medium at each receiver
    r = np.sqrt(((rec - src[:1]) ** 2).sum(1)) + h
    c = 1000.0 * rng.uniform(1.8, 3.0)
    d = (h ** 3 / (4 * math.pi * r))[:, None] * pulse(t[None] - 1 / f0 - r[:, None] / c)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
    return {"src": src, "rec": rec, "wav": dev(wav), "traces": dev(d)}


def _windows(case, seed):
    """Sizes of the shots' windows: between 2/3 and 4/3 of the case's, as drawn from a survey."""
    if case["op"] != "batch":
        return [(case["nx"], case["ny"])]
    rng = np.random.default_rng(20040)       # the same sizes for every seed
    f = rng.uniform(2 / 3, 4 / 3, (case["shots"], 2))
    return [(int(case["nx"] * a), int(case["ny"] * b)) for a, b in f]


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for i, (nx, ny) in enumerate(_windows(case, seed)):
        one = dict(case, nx=nx, ny=ny)
        out.append((one, _model(one, gen), _shot(one, seed * 101 + i, nx, ny)))
    return out


def prepare(case, seed):
    shots = []
    for one, model, shot in _inputs(case, seed):
        prop = wp.Propagator(KIND[one["kind"]], (one["nx"], one["ny"], one["nz"]), one["nbl"], SPACING[one["kind"]],
                             one["so"], one["nt"], model, dt=_dt(one), snap_mode=SNAP[one["snap"]])
        shots.append((prop, shot))
    return case["op"], shots


def run(state):
    op, shots = state
    prop, s = shots[0]
    if op == "forward":
        traces = prop.forward(s["wav"], s["src"], s["rec"])
        return {"traces": traces, "state": prop.get_state(like=traces)}
    if op == "adjoint":
        return prop.adjoint(s["traces"], s["src"], s["rec"])
    if op == "gradient":
        return prop.gradient(s["wav"], s["src"], s["rec"], s["traces"])
    if op == "aniso":
        return prop.gradient_aniso(s["wav"], s["src"], s["rec"], s["traces"])
    cols = [[s[k] for _, s in shots] for k in ("wav", "src", "rec", "traces")]
    return wp.gradient_batch([p for p, _ in shots], *cols)


def work(case):
    """Per time step and point of the computational grid: the wavefield levels a step reads and
    writes and the model, four bytes each; a gradient adds the transposed step, the stored forward
    level and the gradients it adds to (and the second forward step where checkpoints are 16-bit)."""
    kind, op, so = case["kind"], case["op"], case["so"]
    step = {"tti": 44, "elastic": 84, "acoustic": 16, "elastic2d": 52}[kind]
    flop = {"tti": 18 * so + 34, "elastic": 27 * so + 47, "acoustic": 4.5 * so + 3, "elastic2d": 12 * so + 24}[kind]
    image = {"tti": 16, "elastic": 36, "acoustic": 12, "elastic2d": 0}[kind]
    steps = 1.0
    if op in ("gradient", "aniso", "batch"):
        steps = 3.0 if case["snap"] == "bf16" else 2.0
        step = step * steps + image + (32 if op == "aniso" else 0)
        flop = flop * steps * (1.5 if op == "aniso" else 1.0)
    b = case["nbl"]
    cells = sum((nx + 2 * b) * (ny + (0 if kind == "elastic2d" else 2 * b)) * (case["nz"] + 2 * b)
                for nx, ny in _windows(case, 0))
    return {"bytes": float(step) * cells * case["nt"], "flops": float(flop) * cells * case["nt"]}


# ---------------------------------------------------------------------------
# the same calls in 64 bits: the discrete equations step by step in torch, transposes and gradients
# by automatic differentiation
# ---------------------------------------------------------------------------
class _Taps(torch.autograd.Function):
    """sum_i c_i f(x + o_i) along one axis, zero outside the grid."""

    @staticmethod
    def forward(ctx, f, axis, taps):
        ctx.axis, ctx.taps = axis, taps
        return _Taps.apply_to(f, axis, taps)

    @staticmethod
    def apply_to(f, axis, taps):
        out, n = torch.zeros_like(f), f.shape[axis]
        for o, c in taps:
            if abs(o) < n:
                out.narrow(axis, max(0, -o), n - abs(o)).add_(f.narrow(axis, max(0, o), n - abs(o)), alpha=c)
        return out

    @staticmethod
    def backward(ctx, g):
        return _Taps.apply_to(g, ctx.axis, [(-o, c) for o, c in ctx.taps]), None, None


def _weights(so):
    """Taps of the centred first, the two staggered first and the centred second derivative."""
    m = so // 2
    k = np.arange(1, m + 1)
    powers = lambda x, p: np.linalg.solve((2 * x[None, :] ** p[:, None]).astype(float), (p == p[0]) * 1.0)  # noqa: E731
    c = powers(k.astype(float), 2 * np.arange(m) + 1.0)
    b = powers(k - 0.5, 2 * np.arange(m) + 1.0)
    d2 = 2 * powers(k.astype(float), 2 * np.arange(m) + 2.0)
    centred = [(i, w) for i, w in zip(k, c)] + [(-i, -w) for i, w in zip(k, c)]
    plus = [(i, w) for i, w in zip(k, b)] + [(1 - i, -w) for i, w in zip(k, b)]
    minus = [(i - 1, w) for i, w in zip(k, b)] + [(-i, -w) for i, w in zip(k, b)]
    second = [(0, -2 * d2.sum())] + [(i, w) for i, w in zip(k, d2)] + [(-i, w) for i, w in zip(k, d2)]
    return [[(int(o), float(w)) for o, w in t] for t in (centred, plus, minus, second)]


class _Exact:
    def __init__(self, case, model, shot):
        self.case, self.shot, self.h, self.dt = case, shot, SPACING[case["kind"]], _dt(case)
        self.two_d = case["kind"] == "elastic2d"
        n, b = (case["nx"], case["ny"], case["nz"]), case["nbl"]
        pad = (b, 0 if self.two_d else b, b)
        self.shape = tuple(s + 2 * p for s, p in zip(n, pad))
        self.pad, self.n = pad, n
        self.ids = [torch.arange(-p, s + p, device="cuda").clamp(0, s - 1) for s, p in zip(n, pad)]
        self.C, self.P, self.M, self.L = _weights(case["so"])
        self.model = [a.double() for a in model]
        self.src, self.rec = self.points(shot["src"]), self.points(shot["rec"])

    def extend(self, a):
        for axis, i in enumerate(self.ids):
            a = a.index_select(axis, i)
        return a

    def depth(self, axis, half=0.0):
        s = torch.arange(self.shape[axis], device="cuda", dtype=torch.float64) + half
        lo, hi = self.pad[axis], self.pad[axis] + self.n[axis] - 1
        d = torch.where(s < lo, lo - s, torch.where(s > hi, s - hi, torch.zeros_like(s)))
        view = [1, 1, 1]
        view[axis] = -1
        return d.view(view)

    def points(self, xyz):
        """Flat indices and trilinear weights, 8 for each point."""
        s = torch.from_numpy(xyz.astype(np.float64)).cuda() / self.h + torch.tensor(self.pad, device="cuda")
        i = torch.floor(s)
        f, i = s - i, i.long()
        idx, w = [], []
        for k in range(8):
            o = torch.tensor([k >> 2, k >> 1 & 1, k & 1], device="cuda")
            wt = torch.where(o == 1, f, 1 - f).prod(1)
            q = torch.minimum(i + o, torch.tensor(self.shape, device="cuda") - 1)     # weight 0 beyond the grid
            idx.append((q[:, 0] * self.shape[1] + q[:, 1]) * self.shape[2] + q[:, 2])
            w.append(wt)
        return torch.stack(idx, 1), torch.stack(w, 1)

    def sample(self, u):
        return (u.reshape(-1)[self.rec[0]] * self.rec[1]).sum(1)

    def spread(self, q):
        out = torch.zeros(math.prod(self.shape), dtype=torch.float64, device="cuda")
        return out.index_add(0, self.src[0].reshape(-1), (self.src[1] * q[:, None]).reshape(-1)).view(self.shape)

    def d(self, f, axis, taps):
        return _Taps.apply(f, axis, taps)

    def taper(self, hx, hy, hz):
        g = 1.0
        if self.case["nbl"]:
            for axis, half in enumerate((hx, hy, hz)):
                g = g * torch.exp(-(0.015 * self.depth(axis, half)) ** 2)
        return g

    def mean(self, a, *axes):
        """Average over the nodes at i and i + 1 (the last one again at the end) of each axis."""
        for axis in axes:
            n = a.shape[axis]
            nxt = a.index_select(axis, torch.arange(1, n + 1, device="cuda").clamp(max=n - 1))
            a = 0.5 * (a + nxt)
        return a

    def parameters(self):
        """What gradients are taken of, on the physical grid."""
        if self.case["kind"] in ("tti", "acoustic"):
            return [1 / (1000 * self.model[0]) ** 2] + self.model[1:]
        vp, vs, rho = (1000 * a for a in self.model)
        return [rho * (vp * vp - 2 * vs * vs), rho * vs * vs, 1 / rho]

    def damping(self):
        vp = 1000 * self.model[0]
        v = (vp * torch.sqrt(1 + 2 * self.model[1]) if self.case["kind"] == "tti" else vp).max()
        b = self.case["nbl"]
        s0 = 3 * v / (2 * b * self.h) * math.log(1000.0)
        return sum(s0 * (self.depth(a) / b) ** 2 for a in range(3))

    def stepper(self, par):
        dt, h, kind = self.dt, self.h, self.case["kind"]
        if kind in ("tti", "acoustic"):
            m, half = self.extend(par[0]), 0.5 * dt * self.damping()
            A, B = m * (1 + half), m * (1 - half)
        if kind == "acoustic":
            def step(q, u, u0):
                lap = sum(self.d(u, a, self.L) for a in range(3)) / h ** 2
                return ((dt * dt * (lap + self.spread(q)) + 2 * m * u - B * u0) / A, u)
            return step, 2, lambda s: s[0]
        if kind == "tti":
            eps, delta, th, ph = (self.extend(p) for p in par[1:])
            n = [torch.sin(th) * torch.cos(ph), torch.sin(th) * torch.sin(ph), torch.cos(th)]
            c1, c2 = 1 + 2 * eps, torch.sqrt(1 + 2 * delta)

            def step(q, p, r, p0, r0):
                gp, gr = ([self.d(u, a, self.C) / h for a in range(3)] for u in (p, r))
                wp_, wr = (sum(x * y for x, y in zip(n, g)) for g in (gp, gr))
                h0 = sum(self.d(gp[a] - n[a] * wp_, a, self.C) for a in range(3)) / h
                hz = sum(self.d(n[a] * wr, a, self.C) for a in range(3)) / h
                f = dt * dt * self.spread(q)
                return ((dt * dt * (c1 * h0 + c2 * hz) + f + 2 * m * p - B * p0) / A,
                        (dt * dt * (c2 * h0 + hz) + f + 2 * m * r - B * r0) / A, p, r)
            return step, 4, lambda s: s[0]
        lam, mu, b = (self.extend(p) for p in par)
        c, P, M, d, g = dt / h, self.P, self.M, self.d, self.taper
        bx, by, bz = (self.mean(b, a) for a in range(3))
        mxy, mxz, myz = self.mean(mu, 0, 1), self.mean(mu, 0, 2), self.mean(mu, 1, 2)
        o, e = 0.0, 0.5
        if kind == "elastic2d":
            def step(q, vx, vz, txx, tzz, txz):
                f = dt * self.spread(q)
                vx = g(e, o, o) * (vx + c * bx * (d(txx, 0, P) + d(txz, 2, M)))
                vz = g(o, o, e) * (vz + c * bz * (d(txz, 0, M) + d(tzz, 2, P)))
                exx, ezz = d(vx, 0, M), d(vz, 2, M)
                tr = lam * (exx + ezz)
                return (vx, vz, g(o, o, o) * (txx + c * (tr + 2 * mu * exx)) + f,
                        g(o, o, o) * (tzz + c * (tr + 2 * mu * ezz)) + f,
                        g(e, o, e) * (txz + c * mxz * (d(vx, 2, P) + d(vz, 0, P))))
            return step, 5, lambda s: s[2] + s[3]

        def step(q, vx, vy, vz, txx, tyy, tzz, txy, txz, tyz):
            f = dt * self.spread(q)
            vx = g(e, o, o) * (vx + c * bx * (d(txx, 0, P) + d(txy, 1, M) + d(txz, 2, M)))
            vy = g(o, e, o) * (vy + c * by * (d(txy, 0, M) + d(tyy, 1, P) + d(tyz, 2, M)))
            vz = g(o, o, e) * (vz + c * bz * (d(txz, 0, M) + d(tyz, 1, M) + d(tzz, 2, P)))
            exx, eyy, ezz = d(vx, 0, M), d(vy, 1, M), d(vz, 2, M)
            tr, gn = lam * (exx + eyy + ezz), g(o, o, o)
            return (vx, vy, vz, gn * (txx + c * (tr + 2 * mu * exx)) + f, gn * (tyy + c * (tr + 2 * mu * eyy)) + f,
                    gn * (tzz + c * (tr + 2 * mu * ezz)) + f,
                    g(e, e, o) * (txy + c * mxy * (d(vx, 1, P) + d(vy, 0, P))),
                    g(e, o, e) * (txz + c * mxz * (d(vx, 2, P) + d(vz, 0, P))),
                    g(o, e, e) * (tyz + c * myz * (d(vy, 2, P) + d(vz, 1, P))))
        return step, 9, lambda s: s[3] + s[4] + s[5]

    def forward(self, wav, par, keep):
        step, nf, seen = self.stepper(par)
        s = tuple(torch.zeros(self.shape, dtype=torch.float64, device="cuda") for _ in range(nf))
        traces = []
        for n in range(self.case["nt"]):
            traces.append(self.sample(seen(s)))
            s = checkpoint(step, wav[:, n], *s, use_reentrant=False) if keep else step(wav[:, n], *s)
        return torch.stack(traces, 1), s


def exact(case, seed):
    if case["snap"] == "bf16":
        return None                # the 16-bit rounding of the stored levels is the result's error
    one, model, shot = _inputs(case, seed)[0]
    x = _Exact(one, model, shot)
    wav, par = shot["wav"].double(), x.parameters()
    if case["op"] == "forward":
        with torch.no_grad():
            traces, s = x.forward(wav, par, False)
        return {"traces": traces, "state": list(s)}
    if case["op"] == "adjoint":
        wav.requires_grad_()
        traces, _ = x.forward(wav, par, True)
        return torch.autograd.grad(traces, wav, shot["traces"].double())[0]
    wanted = par if case["op"] == "aniso" or case["kind"] == "elastic" else par[:1]
    for p in wanted:
        p.requires_grad_()
    traces, _ = x.forward(wav, par, True)
    J = 0.5 * ((traces - shot["traces"].double()) ** 2).sum()
    grads = [g.detach() for g in torch.autograd.grad(J, wanted)]
    return grads[0] if len(grads) == 1 else torch.stack(grads), float(J)
