"""What the solver is timed on: the calls its users make, from one Hamiltonian on a 64^2
grid to a batch of 64 solves at 256^2 and a 128^3 solve.

A solve is run for a fixed number of PCG iterations per level (``max_iter``; its stopping rule
is the benchmark's and is not met before), so that a pass is the same work each time.  FP64
solves start from a seeded guess, as a user's do.  HYBRID iterations begin where the method
begins them, near a minimum (after the FP64 lead-in, or from a prolonged coarse solution): their
inputs are states that ``_relax`` has brought there, and no further lead-in is asked for.

``exact`` restates the method (preconditioned nonlinear conjugate gradients of arXiv 2602.17950,
Algorithms 1-3) in plain torch, FP64."""
import math

import numpy as np
import torch

from paper_2602_17950_gb300 import Problem, Server
from paper_2602_17950_gb300.gpsoc import apply_h_noalloc

FP64, HYBRID = 0, 2
TOL, RES_TOL = 1e-12, 1e-10        # the benchmark's energy rule; a residual that no case reaches
BENCH_PAR = (0.9, 1.0, 1000.0, -5.0)
DEV = "cuda"


# ----------------------------------------------------------------- the cases
def _case(kind, n, L, batch=1, iters=0, **more):
    c = {"kind": kind, "dim": len(n), "nx": n[0], "ny": n[1], "nz": n[2] if len(n) == 3 else 1,
         "L": float(L), "batch": batch, "iters": iters}
    c.update(more)
    return c


def listed():
    return [
        # H(Phi) alone, for a caller that steps the wave function itself: the smallest call
        dict(_case("operator", (64, 64), 8.0), name="operator-64"),
        # requests of a served bucket, from submission on the host to the last answer
        dict(_case("server", (64, 64), 10.0, 12, 15), name="served-12x64"),
        # axis transforms of a 3D state, there and back
        dict(_case("fft", (128, 128, 128), 8.0), name="fft-128x128x128"),
        # the small plain-PCG workload (64^2, one solve, FP64): launch latency
        dict(_case("solve", (64, 64), 8.0, 1, 31, precision=FP64), name="fp64-64"),
        # the headline's coarsest level, which opens in FP64 from a vortex guess
        dict(_case("solve", (128, 128), 16.0, 1, 31, precision=FP64, strong=True), name="fp64-128"),
        # many initial guesses or parameters at once on a coarse grid, FP64
        dict(_case("solve", (128, 128), 12.0, 16, 15, precision=FP64), name="fp64-16x128"),
        # a 3D solve in an anisotropic box, FP64
        dict(_case("solve", (64, 32, 128), 8.0, 1, 15, precision=FP64, quartic=True), name="fp64-64x32x128"),
        # the headline's coarsest level after the lead-in
        dict(_case("solve", (128, 128), 12.0, 1, 15, precision=HYBRID), name="hybrid-128"),
        # the headline's middle level, where most of its iterations are
        dict(_case("solve", (256, 256), 12.0, 1, 15, precision=HYBRID), name="hybrid-256"),
        # the whole multigrid call of the headline, 128 -> 256 -> 512
        dict(_case("solve", (512, 512), 16.0, 1, 15, precision=HYBRID, levels=3), name="multigrid-512"),
        # the batched parameter sweep
        dict(_case("solve", (256, 256), 12.0, 64, 15, precision=HYBRID), name="hybrid-64x256"),
        # the 3D workload
        dict(_case("solve", (128, 128, 128), 8.0, 1, 15, precision=HYBRID, quartic=True), name="hybrid-128x128x128"),
    ]


def draw(rng):
    """One more case: any of the kinds, grids from 32 to 512 points per axis and ragged ones,
    batches that are no power of two, up to the points of the largest listed case."""
    kind = rng.choice(["operator", "fft", "solve", "solve", "solve", "solve", "server"])
    if kind == "server":
        return _case("server", (rng.choice([32, 64, 128]),) * 2, 10.0, rng.randint(3, 20), 15)
    if kind == "operator":
        dim = rng.choice([2, 2, 3])
        n = [2 ** rng.randint(5, 8) for _ in range(2)] if dim == 2 else [2 ** rng.randint(3, 5) for _ in range(3)]
        most = min(40, 80000 // math.prod(n))
        return _case("operator", n, 8.0, max(1, int(math.exp(rng.uniform(0.0, math.log(most + 0.99))))))
    dim = rng.choice([2, 2, 2, 3])
    hybrid = rng.random() < 0.5
    low, high = (6, 9) if dim == 2 else (5, 7)
    a = rng.randint(low, high)
    b = rng.choice([a, a, rng.randint(low, high)])
    n = [2 ** a, 2 ** b] if dim == 2 else [2 ** a, 2 ** b, 2 ** rng.choice([a, rng.randint(low, high)])]
    while not hybrid and math.prod(n) > 1 << 19:      # FP64 points take several times as long
        n[n.index(max(n))] //= 2
    most = max(1, min(64, (4 << 20) // math.prod(n) // (1 if hybrid else 8)))
    batch = max(1, int(math.exp(rng.uniform(0.0, math.log(most + 0.99)))))
    L = 8.0 if dim == 3 else 12.0
    if kind == "fft":
        return _case("fft", n, L, batch)
    more = {"precision": HYBRID if hybrid else FP64, "quartic": rng.random() < 0.3}
    if rng.random() < 0.25 and min(n) >= 64:
        more["levels"] = 2
    return _case("solve", n, L, batch, rng.choice([7, 15]) if batch * math.prod(n) < 1 << 20 else 7, **more)


def _n(case):
    return tuple(case[k] for k in ("nx", "ny", "nz"))[:case["dim"]]


def _box(case):
    """Half-widths of the box: ragged axes get their share of the points' spacing within limits."""
    return tuple(case["L"] * (1.0 if k == max(_n(case)) else 0.85) for k in _n(case))


def _trap(case):
    g = (1.0, 1.15, 1.6)               # anisotropic: a minimum is not free to turn
    if case.get("quartic"):
        return {"kind": 1, "g": g[:case["dim"]], "quad": 0.0, "quart": 0.05}
    return {"kind": 0, "g": g[:case["dim"]]}


def _params(case, rng):
    if case.get("strong"):
        return [BENCH_PAR] * case["batch"]
    # near a minimum: parameters whose minimum is well separated, so that a state is soon there
    lo, hi = ((0.0, 0.3, 20.0, 1.0), (0.1, 0.6, 100.0, 3.0)) if _relaxed(case) else \
        ((0.0, 0.0, 50.0, -5.0), (0.9, 1.0, 500.0, 5.0))
    return [tuple(float(rng.uniform(a, b)) for a, b in zip(lo, hi)) for _ in range(case["batch"])]


def _relaxed(case):
    return case["kind"] == "server" or case.get("precision") == HYBRID


# ----------------------------------------------------------------- inputs
def _rng(seed):
    return np.random.RandomState(seed % (1 << 31))


def _guess(n, L, batch, rng, vortices=True):
    """Gaussians of random centre, width and phase per component, some times a vortex phase."""
    ax = [torch.arange(k, dtype=torch.float64, device=DEV) * (2 * l / k) - l for k, l in zip(n, L)]
    grid = torch.meshgrid(*ax[::-1], indexing="ij")[::-1]
    out = torch.empty((batch, 3) + n[::-1], dtype=torch.complex128, device=DEV)
    for s in range(batch):
        for c in range(3):
            w, t = rng.uniform(0.8, 1.6), rng.uniform(0.0, 2 * math.pi)
            r2 = sum((x - rng.uniform(-1, 1)) ** 2 for x in grid)
            f = torch.exp(-r2 / (2 * w * w)) * complex(math.cos(t), math.sin(t))
            if vortices and (s + c) % 2:
                f = f * torch.complex(grid[0] - rng.uniform(-1.5, 1.5), grid[1] - rng.uniform(-1.5, 1.5))
            out[s, c] = f / torch.linalg.vector_norm(f)
    return out


def _near_minimum(n, L, pars, trap, rng):
    """States near a minimum on grid n: relaxed on a coarse grid, then carried to n as the
    multigrid does and relaxed a little more."""
    nc = tuple(min(k, 64 if len(n) == 2 else 32) for k in n)
    m = _Model(nc, L, pars, trap)
    psi = _relax(m, _guess(nc, L, len(pars), rng, vortices=False), 300)
    while nc != n:
        nf = tuple(min(2 * a, b) for a, b in zip(nc, n))
        psi = _pad(psi, nc, nf)
        nc = nf
        psi = _relax(_Model(nc, L, pars, trap), psi, 40)
    return psi


def prepare(case, seed):
    rng = _rng(seed)
    n, L, trap, pars = _n(case), _box(case), _trap(case), _params(case, rng)
    kind, B = case["kind"], case["batch"]
    st = {"case": case, "n": n, "L": L, "trap": trap, "pars": pars}
    if kind == "operator":
        st["psi"] = _unit(_guess(n, L, B, rng), n, L)
        st["out"] = torch.empty_like(st["psi"])
        return st
    if kind == "fft":
        st["psi"] = _guess(n, L, B, rng)
        st["work"], st["spec"] = torch.empty_like(st["psi"]), torch.empty_like(st["psi"])
        st["stream"] = torch.cuda.Stream()
        st["problem"] = Problem(n, L, pars, trap=trap, stream=st["stream"].cuda_stream)
        torch.cuda.synchronize()
        return st
    if kind == "server":
        psi = _near_minimum(n, L, pars, trap, rng).cpu().numpy()
        st["requests"] = [np.ascontiguousarray(p) for p in psi]
        st["server"] = Server(hbm_budget_bytes=20e9, slots_per_bucket=16, precision=HYBRID)
        return st
    levels = case.get("levels", 1)
    start = tuple(k >> (levels - 1) for k in n)
    if _relaxed(case):
        st["psi"] = _near_minimum(start, L, pars, trap, rng)
    else:
        st["psi"] = _guess(start, L, B, rng)
    st["out"] = torch.empty((B, 3) + n[::-1], dtype=torch.complex128, device=DEV)
    st["problem"] = Problem(n, L, pars, trap=trap)
    torch.cuda.synchronize()
    return st


# ----------------------------------------------------------------- one pass
def _options(case, precision):
    return dict(precision=precision, tol=TOL, res_tol=RES_TOL, max_iter=case["iters"],
                cm_levels=case.get("levels", 1), check_every=case["iters"] + 1, hybrid_lead_res=-1.0)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "operator":
        obs = apply_h_noalloc(st["n"], st["L"], st["pars"], st["trap"], st["psi"].data_ptr(), st["out"].data_ptr())
        return {"hpsi": st["out"], "obs": obs}
    if kind == "fft":
        p, work, spec, count = st["problem"], st["work"], st["spec"], 3 * case["batch"]
        with torch.cuda.stream(st["stream"]):
            spec.copy_(st["psi"])
            for axis in range(case["dim"]):
                p.fft_axis(spec.data_ptr(), count, axis)
            work.copy_(spec)
            for axis in range(case["dim"]):
                p.fft_axis(work.data_ptr(), count, axis, inverse=True)
        return {"spectrum": spec, "back": work}
    if kind == "server":
        sv, o = st["server"], _options(case, HYBRID)
        o.pop("precision"), o.pop("cm_levels"), o.pop("check_every")
        tickets = [sv.submit(st["n"], st["L"], q, psi, trap=st["trap"], **o)
                   for q, psi in zip(st["pars"], st["requests"])]
        done = [sv.poll(t, timeout_ms=-1) for t in tickets]
        return {"psi": np.stack([d[1] for d in done]), **_scalars([d[0] for d in done])}
    p = st["problem"]
    p.set_initial_device(st["psi"].data_ptr(), level=case.get("levels", 1) - 1)
    res = p.solve(**_options(case, case["precision"]))
    p.psi_to_device(st["out"].data_ptr())
    return {"psi": st["out"], **_scalars(res)}


def _scalars(res):
    return {"energy": np.array([r["energy"] for r in res]), "mu": np.array([r["mu"] for r in res]),
            "mass": np.array([r["mass"] for r in res])}


# ----------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: the states read once and written once.  Operations: the transforms (5 n log2 n
    each; H takes a forward pass, two inverse passes and the rotation's second array, an
    iteration two H and one preconditioner) and about 400 pointwise ones per point."""
    pts = math.prod(_n(case)) * case["batch"]
    logn = sum(math.log2(k) for k in _n(case))
    axis = 5.0 * 3 * pts                       # one transform of every line, per log2 of its length
    h = 4 * axis * logn
    if case["kind"] == "operator":
        return {"bytes": 2 * 48.0 * pts, "flops": h + 150.0 * pts}
    if case["kind"] == "fft":
        return {"bytes": 3 * 48.0 * pts, "flops": 2 * axis * logn}
    per, flops = 2 * h + 2 * axis * logn + 400.0 * pts, 0.0
    for lev in range(case.get("levels", 1)):
        flops += case["iters"] * per / 2 ** (case["dim"] * lev)
    first = 48.0 * pts / 2 ** (case["dim"] * (case.get("levels", 1) - 1))
    return {"bytes": first + 48.0 * pts, "flops": flops}


# ----------------------------------------------------------------- the method in plain torch, 64 bits
def _unit(psi, n, L):
    dV = math.prod(2 * l / k for k, l in zip(n, L))
    mass = (psi.real ** 2 + psi.imag ** 2).sum(dim=tuple(range(1, psi.dim())), keepdim=True) * dV
    return psi / torch.sqrt(mass)


def _pad(psi, nc, nf):
    """Spectral zero padding from grid nc to grid nf."""
    d = len(nc)
    out = torch.zeros(psi.shape[:2] + nf[::-1], dtype=psi.dtype, device=psi.device)
    at = []
    for a, b in zip(nc[::-1], nf[::-1]):
        p = torch.arange(a, device=psi.device)
        at.append(torch.where(p < a // 2, p, p - a) % b if a != b else p)
    axes = tuple(range(2, 2 + d))
    hat = torch.fft.fftn(psi, dim=axes)
    grid = torch.meshgrid(*at, indexing="ij")
    out[(slice(None), slice(None)) + grid] = hat
    return torch.fft.ifftn(out, dim=axes) * (math.prod(nf) / math.prod(nc))


class _Model:
    """Energy, Hamiltonian and preconditioner of a batch of problems on one grid."""

    def __init__(self, n, L, pars, trap):
        self.n, self.d, self.axes = n, len(n), tuple(range(2, 2 + len(n)))
        self.dV = math.prod(2 * l / k for k, l in zip(n, L))
        one = (1,) * self.d

        def along(v, a):                   # a vector over axis a (x, y, z), for the arrays' order z, y, x
            s = list(one)
            s[self.d - 1 - a] = -1
            return v.reshape(s)
        x = [along(torch.arange(k, dtype=torch.float64, device=DEV) * (2 * l / k) - l, a)
             for a, (k, l) in enumerate(zip(n, L))]
        self.k = [along(torch.fft.fftfreq(k, 1.0 / k, dtype=torch.float64, device=DEV) * (math.pi / l), a)
                  for a, (k, l) in enumerate(zip(n, L))]
        self.x, self.y = x[0], x[1]
        r2 = sum(v * v for v in x)
        self.V = sum(0.5 * g * g * v * v for g, v in zip(trap["g"], x))
        if trap["kind"]:
            self.V = self.V + trap["quad"] * r2 + trap["quart"] * r2 * r2
        self.k2 = 0.5 * sum(v * v for v in self.k)
        p = torch.tensor(pars, dtype=torch.float64, device=DEV)
        self.Om, self.ga, self.c0, self.c1 = (p[:, i].reshape((-1,) + one) for i in range(4))

    def fft(self, u):
        return torch.fft.fftn(u, dim=self.axes)

    def ifft(self, u):
        return torch.fft.ifftn(u, dim=self.axes)

    def lin(self, u):
        """The linear part: kinetic, spin-orbit, rotation, trap."""
        h = self.fft(u)
        kx, ky = self.k[0], self.k[1]
        s0, s1 = torch.complex(-kx + 0 * ky, ky + 0 * kx), torch.complex(-kx + 0 * ky, -ky + 0 * kx)
        g = self.ga
        t = torch.stack([self.k2 * h[:, 0] - g * (s0 * h[:, 1]),
                         self.k2 * h[:, 1] - g * (s1 * h[:, 0] + s0 * h[:, 2]),
                         self.k2 * h[:, 2] - g * (s1 * h[:, 1])], dim=1)
        Om = self.Om[:, None]
        ax, ay = 2 + self.d - 1, 2 + self.d - 2
        dx = torch.fft.ifft(kx * torch.fft.fft(u, dim=ax), dim=ax)
        dy = torch.fft.ifft(ky * torch.fft.fft(u, dim=ay), dim=ay)
        return self.ifft(t) + Om * (self.y * dx - self.x * dy) + self.V * u

    @staticmethod
    def spin(u, v):
        """The symmetric cross term of the spin vector of two states: F(u) for u = v."""
        a = 0.5 * (u[:, 1].conj() * v[:, 0] + u[:, 2].conj() * v[:, 1] + v[:, 1].conj() * u[:, 0]
                   + v[:, 2].conj() * u[:, 1])
        z = (u[:, 0].conj() * v[:, 0]).real - (u[:, 2].conj() * v[:, 2]).real
        r = math.sqrt(2.0)
        return torch.stack([r * a.real, -r * a.imag, z], dim=1)

    @staticmethod
    def rho(u, v):
        return (u.real * v.real + u.imag * v.imag).sum(dim=1)

    def interact(self, f, u):
        """c0 rho(f) u + c1 (F(f).f) u, the densities those of f."""
        F = self.spin(f, f)
        m = torch.complex(F[:, 0], -F[:, 1]) / math.sqrt(2.0)      # F_- / sqrt 2
        Fz = F[:, 2]
        w = torch.stack([Fz * u[:, 0] + m * u[:, 1], m.conj() * u[:, 0] + m * u[:, 2],
                         m.conj() * u[:, 1] - Fz * u[:, 2]], dim=1)
        return self.c0[:, None] * self.rho(f, f)[:, None] * u + self.c1[:, None] * w

    def total(self, a):
        return a.sum(dim=tuple(range(1, a.dim()))) * self.dV

    def inner(self, u, v):
        return self.total(u.real * v.real + u.imag * v.imag)

    def observables(self, u, Hl):
        """E, mu, alpha, masses, <H_lin u, u>."""
        Q = self.inner(Hl, u)
        rho, F = self.rho(u, u), self.spin(u, u)
        c0, c1 = self.c0.flatten(), self.c1.flatten()
        I, J = self.total(rho * rho), self.total(F * F)
        m = u.real ** 2 + u.imag ** 2
        h = self.fft(u)
        kin = (self.k2 * (h.real ** 2 + h.imag ** 2)).sum(dim=self.axes) / math.prod(self.n)
        rest = ((self.V + (self.c0 * rho)[:, None]) * m).sum(dim=self.axes)
        return (Q + 0.5 * (c0 * I + c1 * J), Q + c0 * I + c1 * J, (kin + rest) * self.dV,
                m.sum(dim=self.axes) * self.dV, Q, I, J)

    def precondition(self, r, u, alpha):
        al = alpha.reshape(alpha.shape + (1,) * self.d)
        s = torch.rsqrt(torch.maximum(al + self.V + (self.c0 * self.rho(u, u))[:, None], 1e-12 * al))
        return s * self.ifft(self.fft(s * r) / (al + self.k2))


def _pcg(m, u, iters, stop_res=0.0, search=True):
    """`iters` iterations of Algorithms 1 and 2 for every solve (a solve stays where it is once
    its residual is below stop_res); u, E, mu, masses of the last iterate."""
    u = u / torch.sqrt(m.inner(u, u)).reshape((-1,) + (1,) * (m.d + 1))
    col = lambda v: v.reshape((-1,) + (1,) * (m.d + 1))  # noqa: E731
    r_old = P_old = s_old = None
    c0, c1 = m.c0.flatten(), m.c1.flatten()
    for it in range(iters + 1):
        Hl = m.lin(u)
        E, mu, alpha, mass, Q, I0, J0 = m.observables(u, Hl)
        H = Hl + m.interact(u, u)
        r = H - col(mu) * u
        far = r.abs().flatten(1).amax(dim=1) >= stop_res if stop_res else None
        if it == iters or (stop_res and not bool(far.any())):
            break
        amax = alpha.abs().amax(dim=1, keepdim=True)
        z = m.precondition(r, u, torch.maximum(alpha, 1e-12 * amax + 1e-300))
        s = m.inner(r, z)
        D = -z
        if P_old is not None:
            beta = torch.clamp((s - m.inner(r_old, z)) / s_old, min=0.0)
            beta = torch.where(-s + beta * m.inner(r, P_old) < 0, beta, torch.zeros_like(beta))
            D = D + col(beta) * P_old
        P = D - col(m.inner(D, u)) * u
        nP = torch.sqrt(m.inner(P, P))
        p = P / col(nP)
        # E(cos t u + sin t p) - E(u) from the integrals of its explicit form
        lp = m.lin(p)
        R, rp, ru = m.rho(u, p), m.rho(p, p), m.rho(u, u)
        Fu, Fx, Fp = m.spin(u, u), m.spin(u, p), m.spin(p, p)
        T = lambda a, b: m.total(a * b)  # noqa: E731
        I = [I0, T(ru, R), T(ru, rp), T(R, R), T(R, rp), T(rp, rp)]
        J = [J0, T(Fu, Fx), T(Fu, Fp), T(Fx, Fx), T(Fx, Fp), T(Fp, Fp)]
        x, pp = m.inner(Hl, p), m.inner(lp, p)
        a = -mu + pp + c0 * (I[2] + 2 * I[3]) + c1 * (J[2] + 2 * J[3])
        b = 2 * (x + c0 * I[1] + c1 * J[1])

        def change(t):
            sn, cs = torch.sin(t), torch.cos(t)
            f0, f1, f2 = -sn * sn, 2 * sn * cs, sn * sn
            e = f0 * Q + f1 * x + f2 * pp
            for c, K in ((c0, I), (c1, J)):
                l = f0 * K[0] + f1 * K[1] + f2 * K[2]
                q = (f0 * f0 * K[0] + f1 * f1 * K[3] + f2 * f2 * K[5]
                     + 2 * (f0 * f1 * K[1] + f0 * f2 * K[2] + f1 * f2 * K[4]))
                e = e + c * (l + 0.5 * q)
            return e
        t = torch.where(a > 0, -b / (2 * a), torch.full_like(a, 0.1))
        while search:                     # halvings until the energy falls
            bad = change(t) >= 0 if far is None else (change(t) >= 0) & far & (t > 1e-9)
            if not bool(bad.any()):
                break
            t = torch.where(bad, 0.5 * t, t)
        if far is not None:
            t = torch.where(far, t, torch.zeros_like(t))
        r_old, P_old, s_old = r, P, s
        u = col(torch.cos(t)) * u + col(torch.sin(t)) * p
        u = u / torch.sqrt(col(m.inner(u, u)))
    return u, E, mu, mass


def _relax(m, u, iters):
    return _pcg(m, u, iters, stop_res=1e-6, search=False)[0]


def exact(case, seed):
    rng = _rng(seed)
    n, L, trap, pars = _n(case), _box(case), _trap(case), _params(case, rng)
    kind = case["kind"]
    if kind == "operator":
        m = _Model(n, L, pars, trap)
        u = _unit(_guess(n, L, case["batch"], rng), n, L)
        Hl = m.lin(u)
        E, mu, alpha, mass, Q, _, _ = m.observables(u, Hl)
        obs = torch.cat([E[:, None], mu[:, None], alpha, mass, Q[:, None]], dim=1)
        return {"hpsi": Hl + m.interact(u, u), "obs": obs}
    if kind == "fft":
        u = _guess(n, L, case["batch"], rng)
        return {"spectrum": torch.fft.fftn(u, dim=tuple(range(2, u.dim()))), "back": u}
    levels = case.get("levels", 1)
    k = tuple(v >> (levels - 1) for v in n)
    u = _near_minimum(k, L, pars, trap, rng) if _relaxed(case) else _guess(k, L, case["batch"], rng)
    while True:
        u, E, mu, mass = _pcg(_Model(k, L, pars, trap), u, case["iters"])
        if k == n:
            break
        k2 = tuple(2 * v for v in k)
        u, k = _pad(u, k, k2), k2
    return {"psi": u, "energy": E, "mu": mu, "mass": mass}
