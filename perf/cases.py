"""Workloads for timing the library through its Python entry points.

Each case is what a program of one of the library's users does over and over:
apply the operator, apply the preconditioner, solve a batch of wavefields, form
a misfit gradient or a Gauss-Newton product, or serve a stream of requests.
Models are layered media whose velocity rises with depth, with smooth anomalies,
as in the repository's synthetic workloads; every model, source position and
right-hand side follows from the seed.

Wavefield solves run to a relative FP64 residual of 1e-12: the repository's own
parity tests solve to 1e-10 .. 1e-12, and at that depth the refined field does
not depend on the rounding of the complex64 iterations that led to it.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  model, right-hand sides and buffers on the GPU
    run(state)           one pass
    work(case)           bytes and operations one pass cannot do without
    exact(case, seed)    the outputs in 64 bits by plain NumPy
"""
from __future__ import annotations

import numpy as np
import torch

import paper_1712_08743_gb300 as hg
from paper_1712_08743_gb300.autograd import FWIProblem, HelmFWI

TOL = 1e-12
NPML = 20
ALPHA = 0.5
WJ = 0.5           # damped-Jacobi weight of the solver's preconditioner
LAM = 1e-3         # regulariser weight of the misfit


def listed():
    return [
        # one field through the operator on the small plain grid (101 x 101 physical): the smallest
        # call a user makes, for instance a residual check after a solve
        dict(name="apply_c64_101_1rhs", kind="apply", Px=101, Pz=101, h=10.0, f0=5.0, f1=5.0, nf=1, ns=1, prec="fp32"),
        # FP64 operator on a shot gather of the batched grid (64 fields at once): residuals of a whole batch
        dict(name="apply_c128_401x201_64rhs", kind="apply", Px=401, Pz=201, h=10.0, f0=7.0, f1=7.0, nf=1, ns=64,
             prec="fp64"),
        # the preconditioner on its own, as an outer Krylov method of the user's calls it: the single
        # large grid with one vector, and the batched grid with 64 vectors at two frequencies
        dict(name="cycle_1001_1rhs", kind="cycle", Px=1001, Pz=1001, h=5.0, f0=15.0, f1=15.0, nf=1, ns=1),
        dict(name="cycle_401x201_64rhs", kind="cycle", Px=401, Pz=201, h=10.0, f0=4.0, f1=6.0, nf=2, ns=32),
        # the small plain case with the library's defaults, point source in, host field out
        dict(name="solve_101_default", kind="solve", Px=101, Pz=101, h=10.0, f0=5.0, f1=5.0, nf=1, ns=1,
             krylov="bicgstab", prec="mixed", restart=30, reorth="always", inner=1e-2, rhs="point", density=False),
        # odd, unequal sides, five frequencies at once, general right-hand sides on the device, FGMRES defaults
        dict(name="solve_173x97_5f_fields", kind="solve", Px=173, Pz=97, h=10.0, f0=3.0, f1=9.0, nf=5, ns=1,
             krylov="fgmres", prec="mixed", restart=30, reorth="always", inner=1e-2, rhs="field", density=False),
        # the single large solve: 1001 x 1001 at 15 Hz, FGMRES(10) with one Gram-Schmidt pass
        dict(name="solve_1001_fgmres10", kind="solve", Px=1001, Pz=1001, h=5.0, f0=15.0, f1=15.0, nf=1, ns=1,
             krylov="fgmres", prec="mixed", restart=10, reorth="never", inner=5e-2, rhs="field", density=False),
        # the batched workload: 64 shots times 5 frequencies of one model in one call
        dict(name="solve_401x201_320rhs", kind="solve", Px=401, Pz=201, h=10.0, f0=3.0, f1=7.0, nf=5, ns=64,
             krylov="bicgstab", prec="mixed", restart=30, reorth="always", inner=1e-2, rhs="field", density=False),
        # variable density (Eq. 1): four shots, FGMRES(10)
        dict(name="solve_density_301x151_4rhs", kind="solve", Px=301, Pz=151, h=10.0, f0=6.0, f1=6.0, nf=1, ns=4,
             krylov="fgmres", prec="mixed", restart=10, reorth="never", inner=5e-2, rhs="field", density=True),
        # everything in complex128, the plain FP64 mode
        dict(name="solve_fp64_201x151_2rhs", kind="solve", Px=201, Pz=151, h=10.0, f0=6.0, f1=6.0, nf=1, ns=2,
             krylov="bicgstab", prec="fp64", restart=30, reorth="always", inner=1e-2, rhs="field", density=False),
        # one evaluation of the misfit and its gradient through autograd: model set-up, 32 shots times 4
        # frequencies forward, the adjoint solves and the gradient
        dict(name="fwi_401x201_128rhs", kind="fwi", Px=401, Pz=201, h=10.0, f0=3.0, f1=6.0, nf=4, ns=32, nr=201),
        # twelve requests of one shape at once through the serving queue, a model and a frequency each
        dict(name="serve_128_12req", kind="serve", Px=128, Pz=128, h=0.0, f0=5.0, f1=10.0, nf=12, ns=1),
    ]


def _size(rng, lo, hi):
    """log-uniform whole number in [lo, hi]"""
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "cycle", "cycle", "solve", "solve", "solve", "fwi", "serve"])
    hi = {"apply": 1001, "cycle": 1001, "solve": 400, "fwi": 300, "serve": 200}[kind]
    Px, Pz = _size(rng, 48, hi), _size(rng, 48, hi)
    h = rng.choice([5.0, 8.0, 10.0, 12.5])
    # 10 .. 25 nodes per wavelength at 1500 m/s for the highest frequency
    f1 = round(1500.0 / (h * rng.uniform(10.0, 25.0)), 2)
    f0 = round(f1 * rng.uniform(0.5, 0.9), 2)
    n = (Px + 2 * NPML) * (Pz + 2 * NPML)
    cap = {"apply": 12e6, "cycle": 8e6, "solve": 2e6, "fwi": 2e6, "serve": 5e5}[kind]
    most = max(1, min(256, int(cap / n)))
    b = _size(rng, 1, most)
    nf = rng.choice([k for k in (1, 2, 3, 5) if k <= b])
    case = dict(kind=kind, Px=Px, Pz=Pz, h=h, f0=f0, f1=f1, nf=nf, ns=max(1, b // nf))
    if kind == "apply":
        case["prec"] = rng.choice(["fp32", "fp64"])
    elif kind == "solve":
        prec = "fp64" if n * b < 2e5 and rng.random() < 0.4 else "mixed"
        kry = rng.choice(["bicgstab", "fgmres"])
        case.update(krylov=kry, prec=prec, restart=rng.choice([10, 20, 30]),
                    reorth=rng.choice(["always", "never"]), inner=rng.choice([1e-2, 5e-2]),
                    rhs=rng.choice(["point", "field"]), density=rng.random() < 0.25)
    elif kind == "fwi":
        case.update(nr=_size(rng, 8, Px))
    elif kind == "serve":
        case.update(nf=min(b, 12), ns=1, h=0.0)
    return case


# ------------------------------------------------------------------ inputs
def _velocity(rng, Px, Pz, h, vmin=1500.0, vmax=4000.0):
    """A survey area's layered model, velocity rising with depth over a dipping base: the structure is
    the same for every seed, as it is over the iterations of an inversion, while interfaces and
    velocities (by about a per cent) and three smooth anomalies are the seed's own."""
    area = np.random.default_rng(3)
    x, z = np.linspace(0.0, 1.0, Px), np.linspace(0.0, 1.0, Pz)
    X, Z = np.meshgrid(x, z)
    depths = np.sort(area.uniform(0.0, 1.0, 7)) * (1.0 + rng.uniform(-0.01, 0.01, 7))
    vel = np.sort(area.uniform(vmin, vmax, 8)) * (1.0 + rng.uniform(-0.01, 0.01, 8))
    c = vel[np.searchsorted(np.sort(depths), Z)]
    base = area.uniform(0.3, 0.6) + X * np.tan(np.deg2rad(area.uniform(5.0, 20.0))) + rng.uniform(-0.01, 0.01)
    c = np.where(Z > base, np.maximum(c, 3500.0), c)
    for _ in range(3):
        amp, sig = rng.uniform(-100.0, 100.0), rng.uniform(0.03, 0.08)
        cx, cz = rng.uniform(0.1, 0.9), rng.uniform(0.1, 0.9)
        c = c + amp * np.exp(-((X - cx) ** 2 + ((Z - cz) * Pz / Px) ** 2) / (2.0 * sig ** 2))
    return np.clip(c, vmin, vmax + 100.0)


def _inputs(case, seed):
    """Host inputs of a case: everything prepare() uploads and exact() starts from."""
    rng = np.random.default_rng([int(seed), 17])
    Px, Pz = case["Px"], case["Pz"]
    d = {}
    if case["kind"] == "serve":
        # ten nodes per wavelength at 1500 m/s for each request's own frequency
        d["f"] = rng.uniform(case["f0"], case["f1"], case["nf"])
        d["h"] = 1500.0 / (10.0 * d["f"])
        d["c"] = [_velocity(rng, Px, Pz, float(h)) for h in d["h"]]
        d["src"] = np.stack([rng.integers(2, Px - 2, case["nf"]), np.full(case["nf"], min(2, Pz - 1))], 1)
        return d
    h = case["h"]
    d["c"] = _velocity(rng, Px, Pz, h)
    freqs = np.linspace(case["f0"], case["f1"], case["nf"]) if case["nf"] > 1 else np.array([case["f1"]])
    d["freqs"] = 2.0 * np.pi * freqs
    ns = case["ns"]
    lo, hi = 2, Px - 3
    off = rng.uniform(0.0, 1.0)
    sx = np.clip(lo + np.floor((np.arange(ns) + off) * (hi - lo) / ns).astype(int), lo, hi)
    d["shots"] = np.stack([sx, np.full(ns, 2)], 1)
    d["omega"] = np.repeat(d["freqs"], ns)                      # [nf * ns], one per right-hand side
    d["src"] = np.tile(d["shots"], (case["nf"], 1))
    if case.get("density"):
        d["rho"] = 0.31 * d["c"] ** 0.25                         # Gardner's relation
    if case["kind"] == "fwi":
        nr = case["nr"]
        rx = np.floor(np.arange(nr) * (Px - 1) / max(1, nr - 1)).astype(int)
        d["rec"] = np.stack([rx, np.full(nr, 2)], 1)
        # observed data: far-field response of a uniform medium, one velocity per shot
        k = d["freqs"][:, None, None] / rng.uniform(1600.0, 2200.0, ns)[None, :, None]
        r = (np.abs(d["shots"][:, 0][:, None] - rx[None, :]) + 1.0) * h
        d["d_obs"] = np.sqrt(2.0 / (np.pi * k * r[None])) * np.exp(-1j * (k * r[None] + 0.25 * np.pi)) / 4.0
    return d


def _field(case, seed, dtype, device):
    """Random complex vectors [nrhs][nz][nx], drawn on the GPU where there is one."""
    nx, nz, b = case["Px"] + 2 * NPML, case["Pz"] + 2 * NPML, case["nf"] * case["ns"]
    g = torch.Generator(device=device).manual_seed(int(seed) * 7919 + 3)
    return torch.randn((b, nz, nx), dtype=dtype, device=device, generator=g)


def _sources(case, inp, device):
    """Point sources as complex128 fields (a shot's unit source is 1 / h^2 at its node), each shot
    with an amplitude and phase of its own."""
    nx, nz, b = case["Px"] + 2 * NPML, case["Pz"] + 2 * NPML, case["nf"] * case["ns"]
    f = torch.zeros((b, nz, nx), dtype=torch.complex128, device=device)
    at = torch.as_tensor(inp["src"] + NPML, device=device)
    k = torch.arange(b, device=device)
    amp = torch.exp(1j * 0.7 * k.to(torch.float64)).to(torch.complex128) * (1.0 + 0.1 * (k % 5)) / case["h"] ** 2
    f[k, at[:, 1], at[:, 0]] = amp
    return f


def prepare(case, seed):
    inp = _inputs(case, seed)
    kind, dev = case["kind"], torch.device("cuda")
    st = dict(case=case, inp=inp, ctx=hg.Context(0))
    if kind == "serve":
        hg.helm_serve_config(st["ctx"], max_batch=16, max_slots=1)
        st["slow"] = [1.0 / c for c in inp["c"]]
        st["opts"] = dict(tol=TOL, krylov=hg.HELM_KRYLOV_FGMRES, restart=30, reorth=hg.HELM_REORTH_NEVER, max_it=20000)
        return st
    if kind == "fwi":
        st["m"] = torch.tensor(1.0 / inp["c"], dtype=torch.float64, requires_grad=True)
        st["prob"] = FWIProblem(st["ctx"], case["h"], inp["freqs"], inp["shots"], inp["rec"], inp["d_obs"], LAM, NPML,
                                ALPHA, dict(tol=TOL))
        return st
    st["model"] = hg.helm_create_model(st["ctx"], 1.0 / inp["c"], case["h"], NPML, ALPHA, density=inp.get("rho"))
    if kind == "apply":
        st["x"] = _field(case, seed, torch.complex128 if case["prec"] == "fp64" else torch.complex64, dev)
        st["prec"] = hg.HELM_PREC_FP64 if case["prec"] == "fp64" else hg.HELM_PREC_FP32
    elif kind == "cycle":
        st["x"] = _field(case, seed, torch.complex64, dev)
    else:
        st["opts"] = hg.helm_default_opts(
            tol=TOL, precision=case["prec"], restart=case["restart"], inner_tol=case["inner"], max_it=20000,
            krylov=hg.HELM_KRYLOV_FGMRES if case["krylov"] == "fgmres" else hg.HELM_KRYLOV_BICGSTAB,
            reorth=hg.HELM_REORTH_ALWAYS if case["reorth"] == "always" else hg.HELM_REORTH_NEVER)
        if case["rhs"] == "field":
            st["f"] = _sources(case, inp, dev) if case["ns"] > 1 or case["Px"] > 500 else _field(case, seed, torch.complex128, dev)
            st["u"] = torch.empty_like(st["f"])
    return st


def run(st):
    case, inp = st["case"], st["inp"]
    kind = case["kind"]
    if kind == "apply":
        return hg.helm_apply(st["model"], inp["omega"], st["x"], st["prec"])
    if kind == "cycle":
        return hg.helm_vcycle(st["model"], inp["omega"], st["x"], omega_jacobi=WJ)
    if kind == "solve":
        if case["rhs"] == "point":
            return hg.helm_solve(st["model"], inp["omega"], inp["src"], opts=st["opts"])[0]
        return hg.helm_solve(st["model"], inp["omega"], f=st["f"], opts=st["opts"], out=st["u"])[0]
    if kind == "fwi":
        m = st["m"]
        m.grad = None
        J = HelmFWI.apply(m, st["prob"])
        J.backward()
        return dict(J=J.detach(), grad=m.grad)
    ctx = st["ctx"]
    tickets = [hg.helm_submit(ctx, st["slow"][k], float(inp["h"][k]), 2.0 * np.pi * float(inp["f"][k]),
                              inp["src"][k], NPML, ALPHA, st["opts"]) for k in range(case["nf"])]
    out = []
    for t in tickets:
        out.append(hg.helm_poll(ctx, t).u)
        hg.helm_release(ctx, t)
    return out


def work(case):
    """Each input read once and each output written once; for the iterative paths, one application of
    the operator to each field is all the arithmetic that is certain beforehand."""
    n = float((case["Px"] + 2 * NPML) * (case["Pz"] + 2 * NPML))
    b = case["nf"] * case["ns"]
    op = 14.0 * n * b                       # four complex additions and one complex product per node
    if case["kind"] == "apply":
        e = 16.0 if case["prec"] == "fp64" else 8.0
        return dict(bytes=n * (2 * e * b + e / 2), flops=op)
    if case["kind"] == "cycle":
        return dict(bytes=n * (16.0 * b + 4.0), flops=2.0 * op)
    if case["kind"] == "solve":
        return dict(bytes=n * (16.0 * b * (2 if case["rhs"] == "field" else 1) + 8.0 * (2 if case["density"] else 1)),
                    flops=op)
    if case["kind"] == "fwi":
        # the slowness in and the gradient out; the forward fields written and read once, the adjoint fields once
        return dict(bytes=n * (16.0 + 48.0 * b) + 16.0 * b * case["nr"], flops=2.0 * op)
    return dict(bytes=n * b * 24.0, flops=op)


# ------------------------------------------------- the same in 64 bits, by plain NumPy
def _pad(a):
    return np.pad(np.asarray(a, np.float64), NPML, mode="edge")


def _alpha(Px, Pz):
    ix, iz = np.arange(Px + 2 * NPML), np.arange(Pz + 2 * NPML)
    dx = np.maximum(np.maximum(NPML - ix, ix - (NPML + Px - 1)), 0)
    dz = np.maximum(np.maximum(NPML - iz, iz - (NPML + Pz - 1)), 0)
    return ALPHA * (np.maximum(dx[None, :], dz[:, None]) / NPML) ** 2


class _Operator:
    """h^2 B of one frequency: edge coefficients (ones without a density) and the complex mass term."""

    def __init__(self, c, h, omega, rho=None):
        m = _pad(1.0 / c)
        Pz, Px = c.shape
        self.mass = (h * omega * m) ** 2 * (1.0 - 1j * _alpha(Px, Pz))
        nz, nx = m.shape
        r = np.ones((nz, nx)) if rho is None else _pad(rho)
        self.e = 2.0 * r[:, :-1] * r[:, 1:] / (r[:, :-1] + r[:, 1:])   # east edge of each node
        self.n = 2.0 * r[:-1] * r[1:] / (r[:-1] + r[1:])               # edge to the next row
        dg = np.zeros((nz, nx))
        dg[:, :-1] += self.e
        dg[:, 1:] += self.e
        dg[:-1] += self.n
        dg[1:] += self.n
        dg[0] += r[0]
        dg[-1] += r[-1]
        dg[:, 0] += r[:, 0]
        dg[:, -1] += r[:, -1]
        self.diag = dg - self.mass

    def apply(self, u):
        y = self.diag * u
        y[..., :, :-1] -= self.e * u[..., :, 1:]
        y[..., :, 1:] -= self.e * u[..., :, :-1]
        y[..., :-1, :] -= self.n * u[..., 1:, :]
        y[..., 1:, :] -= self.n * u[..., :-1, :]
        return y

    def factor(self):
        """Block elimination by rows of the grid (by columns where those are shorter)."""
        self.flip = self.diag.shape[1] > self.diag.shape[0]
        dg = self.diag.T if self.flip else self.diag
        along = self.n.T if self.flip else self.e       # couplings inside a block
        self.cross = self.e.T if self.flip else self.n  # couplings to the next block
        nb, w = dg.shape
        self.inv = np.empty((nb, w, w), np.complex128)
        i = np.arange(w)
        for k in range(nb):
            S = np.zeros((w, w), np.complex128)
            S[i, i] = dg[k]
            S[i[:-1], i[1:]] = -along[k]
            S[i[1:], i[:-1]] = -along[k]
            if k:
                R = self.cross[k - 1]
                S -= R[:, None] * self.inv[k - 1] * R[None, :]
            self.inv[k] = np.linalg.inv(S)
        return self

    def _sweep(self, f):
        g = f.transpose(2, 1, 0) if self.flip else f.transpose(1, 2, 0)     # [block][node][rhs]
        y = np.empty(g.shape, np.complex128)
        nb = len(g)
        for k in range(nb):
            t = g[k] if k == 0 else g[k] + self.cross[k - 1][:, None] * y[k - 1]
            y[k] = self.inv[k] @ t
        for k in range(nb - 2, -1, -1):
            y[k] += self.inv[k] @ (self.cross[k][:, None] * y[k + 1])
        return y.transpose(2, 1, 0) if self.flip else y.transpose(2, 0, 1)

    def solve(self, f):
        u = self._sweep(f)
        for _ in range(2):
            u = u + self._sweep(f - self.apply(u))
        return u


def _prolong(e, nz, nx):
    def one(a, n):      # along the last axis: coarse node I sits on fine node 2I + 1
        out = np.zeros(a.shape[:-1] + (n + 2,), a.dtype)
        out[..., 2:2 + 2 * a.shape[-1]:2] = a
        out[..., 1:1 + 2 * a.shape[-1]:2] += 0.5 * a
        out[..., 3:3 + 2 * a.shape[-1]:2] += 0.5 * a[..., : (n + 2 - 3 + 1) // 2]
        return out[..., 1:n + 1]

    return one(one(e, nx).swapaxes(-1, -2), nz).swapaxes(-1, -2)


def _restrict(r):
    def one(a):
        n = a.shape[-1]
        nc = n // 2
        out = a[..., 1:2 * nc:2] + 0.5 * a[..., 0:2 * nc:2]
        right = a[..., 2:2 * nc + 1:2]
        out[..., :right.shape[-1]] += 0.5 * right
        return out

    return one(one(r).swapaxes(-1, -2)).swapaxes(-1, -2)


def _stencil(M, u):
    """y = M u, M [9][nz][nx] (south-west .. north-east, x fastest)."""
    v = np.pad(u, [(0, 0)] * (u.ndim - 2) + [(1, 1), (1, 1)])
    nz, nx = u.shape[-2:]
    return sum(M[3 * (dz + 1) + dx + 1] * v[..., 1 + dz:1 + dz + nz, 1 + dx:1 + dx + nx]
               for dz in (-1, 0, 1) for dx in (-1, 0, 1))


def _galerkin(M):
    """P^T M P as a 9-point stencil, by probing with the nine 3 x 3 colours."""
    nz, nx = M.shape[1:]
    cz, cx = nz // 2, nx // 2
    K, I = np.meshgrid(np.arange(cz), np.arange(cx), indexing="ij")
    out = np.zeros((9, cz, cx), M.dtype)
    for p in range(3):
        for q in range(3):
            v = ((K % 3 == p) & (I % 3 == q)).astype(M.dtype)
            w = _restrict(_stencil(M, _prolong(v, nz, nx)))
            for dz in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    at = ((K + dz) % 3 == p) & ((I + dx) % 3 == q)
                    out[3 * (dz + 1) + dx + 1][at] = w[at]
    return out


def _dense(M):
    nz, nx = M.shape[1:]
    A = np.zeros((nz, nx, nz, nx), M.dtype)
    for iz in range(nz):
        for ix in range(nx):
            for dz in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    if 0 <= iz + dz < nz and 0 <= ix + dx < nx:
                        A[iz, ix, iz + dz, ix + dx] = M[3 * (dz + 1) + dx + 1][iz, ix]
    return A.reshape(nz * nx, nz * nx)


class _Cycle:
    """One preconditioner application: V-cycle, F-cycle from level lf, damped Jacobi, Galerkin levels,
    an exact solve at level `last` (batches of at most 16: the first of at most 1200 nodes)."""

    def __init__(self, c, h, omega, lf_omega, nrhs):
        m2 = _pad(1.0 / c) ** 2
        hw = (h * omega) ** 2
        nz, nx = m2.shape
        M = np.zeros((9, nz, nx), np.complex128)
        M[4] = 4.0 - hw * (1.0 - 0.5j) * m2
        M[1], M[3], M[5], M[7] = -1.0, -1.0, -1.0, -1.0
        shapes = [(nz, nx)]
        while shapes[-1][0] * shapes[-1][1] > 128 and min(shapes[-1]) >= 4:
            shapes.append((shapes[-1][0] // 2, shapes[-1][1] // 2))
        size = [a * b for a, b in shapes]
        self.last = next(l for l in range(1, len(size)) if size[l] <= 1200) if nrhs <= 16 else len(size) - 1
        cap = next((l for l in range(1, len(size)) if size[l] <= 24576), len(size) - 1)
        self.lf = next((l for l in range(1, cap) if h * lf_omega * 2.0 ** l / c.min() >= 0.7), cap)
        self.M = [M]
        for _ in range(self.last):
            self.M.append(_galerkin(self.M[-1]))
        self.A = _dense(self.M[-1])

    def at(self, f, l, full):
        M = self.M[l]
        nz, nx = M.shape[1:]
        if l == self.last:
            return np.linalg.solve(self.A, f.reshape(len(f), -1).T).T.reshape(f.shape)
        D = M[4]
        u = WJ * f / D
        u = u + _prolong(self.at(_restrict(f - _stencil(M, u)), l + 1, full or l + 1 == self.lf), nz, nx)
        if full:
            u = u + _prolong(self.at(_restrict(f - _stencil(M, u)), l + 1, False), nz, nx)
        return u + WJ * (f - _stencil(M, u)) / D


def exact(case, seed):
    inp = _inputs(case, seed)
    kind, ns = case["kind"], case["ns"]
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if kind == "serve":
        out = []
        for k in range(case["nf"]):
            op = _Operator(inp["c"][k], inp["h"][k], 2.0 * np.pi * inp["f"][k])
            f = np.zeros((1,) + op.diag.shape, np.complex128)
            f[0, inp["src"][k][1] + NPML, inp["src"][k][0] + NPML] = 1.0
            out.append(op.factor().solve(f)[0])
        return out
    h, rho = case["h"], inp.get("rho")
    if kind == "apply":
        x = _field(case, seed, torch.complex128 if case["prec"] == "fp64" else torch.complex64, dev).cpu().numpy()
        op = _Operator(inp["c"], h, 1.0)
        y = np.empty(x.shape, np.complex128)
        unit = op.mass
        for k, w in enumerate(inp["freqs"]):
            op.diag = 4.0 - w * w * unit
            y[k * ns:(k + 1) * ns] = op.apply(x[k * ns:(k + 1) * ns].astype(np.complex128)) / (h * h)
        return y
    if kind == "cycle":
        x = _field(case, seed, torch.complex64, dev).cpu().numpy().astype(np.complex128)
        z = np.empty_like(x)
        for k, w in enumerate(inp["freqs"]):
            cyc = _Cycle(inp["c"], h, w, inp["freqs"].min(), len(x))
            z[k * ns:(k + 1) * ns] = cyc.at(x[k * ns:(k + 1) * ns], 0, False)
        return z
    # a block elimination of grids this large takes longer than it is worth
    short, long = sorted((case["Px"] + 2 * NPML, case["Pz"] + 2 * NPML))
    if short > 500 or case["nf"] * long * (short / 240.0) ** 3 > 2500:
        return None if kind == "solve" else dict(J=None, grad=None)
    if kind == "solve":
        if case["rhs"] == "point":
            f = np.zeros((case["nf"] * ns, case["Pz"] + 2 * NPML, case["Px"] + 2 * NPML), np.complex128)
            f[np.arange(len(f)), inp["src"][:, 1] + NPML, inp["src"][:, 0] + NPML] = 1.0 / (h * h)
        elif ns > 1 or case["Px"] > 500:
            f = _sources(case, inp, dev).cpu().numpy()
        else:
            f = _field(case, seed, torch.complex128, dev).cpu().numpy()
        u = np.empty_like(f)
        for k, w in enumerate(inp["freqs"]):
            op = _Operator(inp["c"], h, w, rho).factor()
            u[k * ns:(k + 1) * ns] = op.solve(h * h * f[k * ns:(k + 1) * ns])
        return u
    # misfit and gradient
    Pz, Px = inp["c"].shape
    nz, nx = Pz + 2 * NPML, Px + 2 * NPML
    m = 1.0 / inp["c"]
    a = _alpha(Px, Pz)
    rec = inp["rec"] + NPML
    J, g = 0.0, np.zeros((nz, nx))
    for k, w in enumerate(inp["freqs"]):
        op = _Operator(inp["c"], h, w).factor()
        f = np.zeros((ns, nz, nx), np.complex128)
        f[np.arange(ns), inp["shots"][:, 1] + NPML, inp["shots"][:, 0] + NPML] = 1.0
        u = op.solve(f)
        r = u[:, rec[:, 1], rec[:, 0]] - inp["d_obs"][k]
        J += float(np.sum(np.abs(r) ** 2))
        q = np.zeros_like(f)
        for s in range(ns):
            np.add.at(q[s], (rec[:, 1], rec[:, 0]), h * h * np.conj(r[s]))
        g += 4.0 * w * w * _pad(m) * np.sum(np.real((1.0 - 1j * a) * u * op.solve(q)), axis=0)
    pz = np.clip(np.arange(nz) - NPML, 0, Pz - 1)
    px = np.clip(np.arange(nx) - NPML, 0, Px - 1)
    grad = np.zeros((Pz, Px))
    np.add.at(grad, (pz[:, None], px[None, :]), g)
    return dict(J=np.array(J + LAM * np.sum(m ** 2)), grad=grad + 2.0 * LAM * m)
