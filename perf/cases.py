"""Performance cases of the implicit SPH thermal-radiative-transfer library.

A case is one pass of what a user's program does with the library, through the
Python binding of the C ABI: whole jobs (set the particles, advance some time
steps, read the energies back), problems whose particles move, batches of small
problems and a served stream of requests.  Inputs are jittered lattices with
ghost layers and the analytic fields of the repository's workloads, made on the
GPU from the seed.

  listed()            the cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) the inputs and the handle a program keeps
  run(state)          one pass; returns e and E of every particle (caller order)
  work(case)          bytes and operations one pass cannot do without
  exact(case, seed)   the same results from 64-bit torch, iterated to rounding
"""
import math

import numpy as np
import torch

from paper_2001_11606_gb300 import sphrt

INTERIOR, DIRICHLET, COPY = 0, 1, 2
WENDLAND = 1
F64 = torch.float64

# the cgs travelling-cosine problem: a = 4 sigma_SB / c, c, k_B / ((gamma - 1) m_p)
CGS_A = 4.0 * 5.670374419e-5 / 2.99792458e10
CGS_C = 2.99792458e10
CGS_CV = 1.380649e-16 / ((5.0 / 3.0 - 1.0) * 1.67262192369e-24)


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _job(problem, nx, ny, nz, steps, mixed=False, post=1, precond="amg", name=None):
    case = dict(kind="job", problem=problem, nx=nx, ny=ny, nz=nz, steps=steps, mixed=mixed,
                post=post, precond=precond)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest problem: launches and host round trips count
        _job("mms", 32, 32, 0, 10, name="mms2d-32"),
        # an ordinary 2-D problem of odd, unequal sides
        _job("mms", 301, 287, 0, 10, name="mms2d-301x287"),
        # temperature-dependent opacity and the Levermore limiter, symmetric V-cycle
        _job("mms-lp", 64, 64, 64, 50, name="mms3d-lp-64"),
        # the library's large FP64 problem, V-cycle-product CG, ragged
        _job("mms", 97, 96, 91, 12, post=0, name="mms3d-97-fp64"),
        # the headline problem, mixed precision, V-cycle-product CG
        _job("mms", 128, 128, 128, 25, mixed=True, post=0, name="mms3d-128-mixed"),
        # dense opaque sphere in a thin medium, mixed precision, odd sides
        _job("sphere", 111, 111, 109, 10, mixed=True, post=0, name="sphere-111-mixed"),
        # the paper's own discretisation: Wendland C4, ~250 neighbours, Larsen
        # limiter, scattering, periodic copy ghosts
        _job("cgs", 40, 40, 40, 10, name="cgs3d-40"),
        # a large request of the serving stream alone: 2-D heating wave between
        # reflecting faces
        _job("wave", 1000, 250, 0, 20, name="wave2d-250k"),
        # adapted smoothing lengths and particles that move every step
        dict(name="moving-40", kind="moving", nx=40, ny=37, nz=33, steps=4),
        # many small problems in one persistent launch per step
        dict(name="batch2d-96", kind="batch", dim=2, count=96, nmin=1000, nmax=20000, steps=20),
        dict(name="batch3d-96", kind="batch", dim=3, count=96, nmin=1000, nmax=20000, steps=20),
        # a stream of uneven requests, 2-D and 3-D, small ones fused
        dict(name="serve-20", kind="serve", count=20, nmin=1000, nmax=120000, steps=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["job"] * 7 + ["moving", "batch", "batch", "serve"])
    if kind == "moving":
        n = [_log_int(rng, 10, 44) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], steps=rng.randint(2, 5))
    if kind == "batch":
        lo = _log_int(rng, 300, 3000)
        return dict(kind=kind, dim=rng.choice([2, 3]), count=_log_int(rng, 4, 128), nmin=lo,
                    nmax=_log_int(rng, lo, 20000), steps=rng.randint(5, 25))
    if kind == "serve":
        lo = _log_int(rng, 300, 5000)
        return dict(kind=kind, count=rng.randint(3, 20), nmin=lo, nmax=_log_int(rng, 2 * lo, 120000),
                    steps=rng.randint(5, 20))
    problem = rng.choice(["mms", "mms", "mms-lp", "sphere", "cgs", "wave"])
    mixed = rng.random() < 0.4
    post = rng.choice([0, 1])
    precond = rng.choice(["amg"] * 8 + ["jacobi", "chebyshev"])
    dim = 3 if problem == "sphere" else rng.choice([2, 3, 3])
    if dim == 2:
        n = [_log_int(rng, 20, 700) for _ in range(2)] + [0]
    else:
        top = 44 if problem == "cgs" else 100
        m = _log_int(rng, 10, top)
        n = [max(8, int(m * rng.uniform(0.85, 1.15))) for _ in range(3)]
    if problem == "wave":  # a slab four times as long as wide
        side = max(6, n[1] // 3)
        n = [4 * side, side, side if dim == 3 else 0]
    cells = n[0] * n[1] * max(1, n[2])
    return _job(problem, n[0], n[1], n[2], min(25, max(3, int(1.2e7 / cells))), mixed, post,
                precond)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rand(seed, k, n, dev):
    g = torch.Generator(device=dev)
    g.manual_seed((int(seed) * 1000003 + k) % (1 << 62))
    return torch.rand(n, generator=g, device=dev, dtype=F64)


def _lattice(counts, dx, seed, layers, faces, dev, jitter=0.1):
    """Jittered lattice with `layers` ghost layers, x fastest.  faces[d]: 'dirichlet',
    'reflect' or 'periodic'; a ghost outside faces of both kinds is Dirichlet."""
    dim = len(counts)
    ext = [c + 2 * layers for c in counts]
    n = math.prod(ext)
    lin = torch.arange(n, device=dev)
    idx = []
    for d in range(dim):
        idx.append(lin % ext[d] - layers)
        lin = lin // ext[d]
    idx = torch.stack(idx, 1)
    u = _rand(seed, 1, n * dim, dev).reshape(n, dim)
    pos = (idx.to(F64) + 0.5 + jitter * (2.0 * u - 1.0)) * dx
    cnt = torch.tensor(counts, device=dev)
    lo, hi = idx < 0, idx >= cnt
    out = lo | hi
    dirichlet = torch.zeros(n, dtype=torch.bool, device=dev)
    copied = torch.zeros(n, dtype=torch.bool, device=dev)
    for d in range(dim):
        if faces[d] == "dirichlet":
            dirichlet |= out[:, d]
        else:
            copied |= out[:, d]
    copied &= ~dirichlet
    kind = torch.zeros(n, dtype=torch.int32, device=dev)
    kind[dirichlet] = DIRICHLET
    kind[copied] = COPY
    copy_of = torch.full((n,), -1, dtype=torch.int64, device=dev)
    if bool(copied.any()):
        src = idx.clone()
        for d in range(dim):
            if faces[d] == "reflect":
                src[:, d] = torch.where(lo[:, d], -1 - src[:, d], src[:, d])
                src[:, d] = torch.where(hi[:, d], 2 * counts[d] - 1 - src[:, d], src[:, d])
            elif faces[d] == "periodic":
                src[:, d] = src[:, d] % counts[d]
        s = torch.zeros(n, dtype=torch.int64, device=dev)
        for d in reversed(range(dim)):
            s = s * ext[d] + src[:, d] + layers
        copy_of = torch.where(copied, s, copy_of)
        at = pos[torch.where(copied, s, torch.arange(n, device=dev))]
        for d in range(dim):
            size = counts[d] * dx
            if faces[d] == "reflect":
                at[:, d] = torch.where(lo[:, d], -at[:, d], at[:, d])
                at[:, d] = torch.where(hi[:, d], 2.0 * size - at[:, d], at[:, d])
            elif faces[d] == "periodic":
                at[:, d] = torch.where(lo[:, d], at[:, d] - size, at[:, d])
                at[:, d] = torch.where(hi[:, d], at[:, d] + size, at[:, d])
        pos = torch.where(copied[:, None], at, pos)
    return dict(dim=dim, counts=tuple(counts), ext=tuple(ext), layers=layers, dx=dx, jitter=jitter,
                pos=pos.contiguous(), kind=kind, copy_of=copy_of)


def _limiter(R, limiter):
    """lambda(R) and its slope: Fick, Levermore, Larsen with k = 2."""
    if limiter == 1:
        den = 6.0 + 3.0 * R + R * R
        return (2.0 + R) / den, -R * (4.0 + R) / (den * den)
    if limiter == 2:
        s = 9.0 + R * R
        return s ** -0.5, -R * s ** -1.5
    return torch.full_like(R, 1.0 / 3.0), torch.zeros_like(R)


def _wave_products(c, s, sign):
    """Gradient and Hessian factors of prod_a cos-like waves: g_a = sign s_a prod_{b!=a} c_b
    and H_ab for unit wave number (c' = sign s, s' = -sign c)."""
    dim = c.shape[1]

    def rest(skip):
        out = torch.ones_like(c[:, 0])
        for a in range(dim):
            if a not in skip:
                out = out * c[:, a]
        return out

    prod = rest(())
    g = torch.stack([sign * s[:, a] * rest((a,)) for a in range(dim)], 1)
    H = [[-prod if a == b else s[:, a] * s[:, b] * rest((a, b)) for b in range(dim)]
         for a in range(dim)]
    return prod, g, H


class _Manufactured:
    """T = 1 + exp(-t)/2 prod sin(pi x_a), E = T^4, e = T; sigma = T^p, D = lambda(R)/sigma."""

    def __init__(self, x, p, limiter):
        self.p, self.limiter = p, limiter
        self.S, g, H = _wave_products(torch.sin(math.pi * x), torch.cos(math.pi * x), 1.0)
        self.g = math.pi * g
        self.lap = -x.shape[1] * math.pi ** 2 * self.S
        self.gn = self.g.norm(dim=1)
        Hg = torch.stack([sum(H[a][b] * self.g[:, b] for b in range(x.shape[1]))
                          for a in range(x.shape[1])], 1) * math.pi ** 2
        self.dgn = torch.where(self.gn[:, None] > 0, Hg / self.gn.clamp_min(1e-300)[:, None],
                               torch.zeros_like(Hg))

    def fields(self, t):
        T = 1.0 + 0.5 * math.exp(-t) * self.S
        return T, T ** 4

    def sources(self, t):
        A = 0.5 * math.exp(-t)
        T, dT = 1.0 + A * self.S, -A * self.S
        sig = T ** self.p
        R = 4.0 * A * self.gn / (sig * T)
        lam, dlam = _limiter(R, self.limiter)
        D = lam / sig
        flux = D * 4.0 * (3.0 * T ** 2 * (A * self.gn) ** 2 + T ** 3 * A * self.lap)
        if self.limiter or self.p:
            q = self.p + 1.0
            dR = 4.0 * (A * self.dgn * (T ** -q)[:, None]
                        - (q * A * self.gn * T ** (-q - 1.0))[:, None] * A * self.g)
            dD = (dlam[:, None] * dR - (lam * self.p / T)[:, None] * A * self.g) / sig[:, None]
            flux = flux + (dD * 4.0 * (T ** 3)[:, None] * A * self.g).sum(1)
        return dT, 4.0 * T ** 3 * dT - flux


class _Cosines:
    """The cgs travelling cosines: e = e0 (1.2 + prod cos k(x - vt)),
    E = E0 (1.2 + prod cos(k(x + vt) - 1/16)), absorption 0.05, scattering 0.95."""

    e0, v, size, sa, ss = 1e13, 5e9, 5.0, 0.05, 0.95

    def __init__(self, x):
        self.x, self.k = x, 2.0 * math.pi / self.size
        self.E0 = 7.0 * CGS_A * (self.e0 / CGS_CV) ** 4

    def _waves(self, t):
        u = self.k * (self.x - self.v * t)
        w = self.k * (self.x + self.v * t) - 1.0 / 16.0
        return (_wave_products(torch.cos(u), torch.sin(u), -1.0),
                _wave_products(torch.cos(w), torch.sin(w), -1.0))

    def fields(self, t):
        (pe, _, _), (pE, _, _) = self._waves(t)
        return self.e0 * (1.2 + pe), self.E0 * (1.2 + pE)

    def sources(self, t):
        (pe, ge, _), (pE, gE, H) = self._waves(t)
        dim, k = self.x.shape[1], self.k
        e, E = self.e0 * (1.2 + pe), self.E0 * (1.2 + pE)
        de = -self.e0 * k * self.v * ge.sum(1)
        dE = self.E0 * k * self.v * gE.sum(1)
        g = self.E0 * k * gE
        gn = g.norm(dim=1)
        Hg = torch.stack([sum(H[a][b] * g[:, b] for b in range(dim)) for a in range(dim)], 1)
        Hg = Hg * self.E0 * k * k
        st = self.sa + self.ss
        R = gn / (st * E)
        lam, dlam = _limiter(R, 2)
        dR = (Hg / gn.clamp_min(1e-300)[:, None] / E[:, None] - (gn / E ** 2)[:, None] * g) / st
        flux = CGS_C / st * ((dlam[:, None] * dR * g).sum(1)
                             + lam * -dim * self.E0 * k * k * pE)
        couple = CGS_C * self.sa * (E - CGS_A * (e / CGS_CV) ** 4)
        return de - couple, dE - flux + couple


def _problem(case, seed, dev):
    """Particles, physics, initial state and per-step inputs of a job or moving case."""
    counts = [c for c in (case["nx"], case["ny"], case["nz"]) if c]
    dim = len(counts)
    problem = case.get("problem", "moving")
    phys = dict(dim=dim, kernel=0, a=1.0, c=1.0, cv=1.0, limiter=0, larsen_k=2.0, opacity_exp=0.0,
                sigma_s=0.0, tol_outer_e=1e-8, tol_outer_E=1e-8, tol_inner_e=1e-13,
                tol_krylov=1e-12, max_outer=50)
    faces, layers, dx, h, dt = ["dirichlet"] * dim, 3, 1.0 / max(counts), 1.5, 1e-3
    if problem == "mms-lp":
        phys.update(limiter=1, opacity_exp=-3.0)
    elif problem == "sphere":
        phys.update(limiter=1)
        dt = 1e-4
    elif problem == "cgs":
        phys.update(kernel=WENDLAND, a=CGS_A, c=CGS_C, cv=CGS_CV, limiter=2,
                    sigma_s=_Cosines.ss, tol_inner_e=1e-12)
        # one period along every axis: unequal sides take the first one's spacing
        faces, layers, h, dx = ["periodic"] * dim, 4, 4.0, _Cosines.size / counts[0]
        counts = [counts[0]] * dim
        dt = _Cosines.size / _Cosines.v / 1000.0
    elif problem == "wave":
        phys.update(limiter=1, opacity_exp=-3.0, max_outer=1000)
        faces, dx, dt = ["dirichlet"] + ["reflect"] * (dim - 1), 1.0 / counts[1], 1e-5
    elif problem == "moving":
        phys.update(kernel=WENDLAND, limiter=2)
        layers, h = 5, 4.0
    L = _lattice(counts, dx, seed, layers, faces, dev)
    x, n = L["pos"], L["pos"].shape[0]
    one = torch.ones(n, dtype=F64, device=dev)
    rho, sigma0, field = one.clone(), one.clone(), None
    if problem in ("mms", "mms-lp", "moving"):
        field = _Manufactured(x, phys["opacity_exp"], phys["limiter"])
        e, E = field.fields(0.0)
    elif problem == "cgs":
        sigma0 = one * _Cosines.sa
        field = _Cosines(x)
        e, E = field.fields(0.0)
    elif problem == "sphere":
        inside = ((x - 0.5) ** 2).sum(1).sqrt() < 0.25
        rho = torch.where(inside, 10.0, 1.0).to(F64)
        sigma0 = torch.where(inside, 1e3, 1.0).to(F64)
        e = torch.where(inside, 1.0, 0.01).to(F64)
        E = e ** 4
    else:
        sigma0 = one * math.exp(float(_rand(seed, 2, 1, dev)) * math.log(100.0))
        e = torch.where((x[:, 0] < 0) & (L["kind"] != COPY), 1.0, 1e-3).to(F64)
        E = e ** 4
    ins = []
    for k in range(1, case["steps"] + 1):
        ins.append((None, None, None, None) if field is None
                   else tuple(v.contiguous() for v in (*field.sources(k * dt),
                                                       *field.fields(k * dt))))
    moves = []
    if problem == "moving":
        moves = [_lattice(counts, dx, seed + 7919 * k, layers, faces, dev)["pos"]
                 for k in range(1, case["steps"])]
    return dict(lattice=L, phys=phys, dt=dt, h=h * dx * one, rho=rho, mass=rho * dx ** dim,
                sigma0=sigma0, e=e.contiguous(), E=E.contiguous(), inputs=ins, moves=moves)


def _small_waves(case, seed, dev):
    """The small heating-wave problems of a batch or a stream: sizes spread log-uniformly over
    [nmin, nmax] and dimensions mixed by the case alone, opacities and lattices by the seed."""
    out = []
    for k in range(case["count"]):
        a, b = (0.5 + k * 0.6180339887) % 1.0, (0.5 + k * 0.7548776662) % 1.0
        dim = case["dim"] if "dim" in case else (2 if b < 0.5 else 3)
        n = math.exp(math.log(case["nmin"]) + a * math.log(case["nmax"] / case["nmin"]))
        side = max(2, round((n / 4.0) ** (1.0 / dim)))
        c = dict(problem="wave", nx=4 * side, ny=side, nz=side if dim == 3 else 0,
                 steps=case["steps"])
        out.append(_problem(c, seed * 4099 + k, dev))
    return out


class _Arrays:
    """Host arrays of one problem, as the batch and the server take them."""

    def __init__(self, p):
        L = p["lattice"]
        self.pos, self.kind, self.copy_of = L["pos"].numpy(), L["kind"].numpy(), L["copy_of"].numpy()
        self.mass, self.rho = p["mass"].numpy(), p["rho"].numpy()
        self.h, self.sigma0 = p["h"].numpy(), p["sigma0"].numpy()
        self.e, self.E = p["e"].numpy(), p["E"].numpy()


PRECOND = {"amg": sphrt.PRECOND_AMG, "jacobi": sphrt.PRECOND_JACOBI,
           "chebyshev": sphrt.PRECOND_CHEBYSHEV}


def prepare(case, seed):
    if case["kind"] in ("batch", "serve"):
        problems = _small_waves(case, seed, "cpu")
        arrays = [_Arrays(p) for p in problems]
        cfgs = [sphrt.config_from_params(p["phys"]) for p in problems]
        state = dict(kind=case["kind"], steps=case["steps"], dt=problems[0]["dt"], arrays=arrays,
                     cfgs=cfgs)
        if case["kind"] == "batch":
            state["batch"] = sphrt.Batch(cfgs[0])
            state["batch"].add_many([(a, a.e, a.E) for a in arrays], threads=4)
        else:
            state["server"] = sphrt.Server()
        return state
    dev = torch.device("cuda")
    p = _problem(case, seed, dev)
    over = {}
    if case["kind"] == "job":
        over = dict(precision=sphrt.MIXED if case["mixed"] else sphrt.FP64,
                    fine_post_smooth=case["post"], precond=PRECOND[case["precond"]],
                    reliable_drop=1e-6)
        if case["precond"] == "chebyshev":
            over.update(cheb_degree=3, fine_post_smooth=1)
    solver = sphrt.Solver(sphrt.config_from_params(p["phys"], **over))
    p.update(kind=case["kind"], solver=solver, e_out=torch.empty_like(p["e"]),
             E_out=torch.empty_like(p["E"]))
    torch.cuda.synchronize()  # the inputs were made on torch's stream
    return p


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _ptr(t):
    return 0 if t is None else t.data_ptr()


def run(state):
    if state["kind"] == "batch":
        b = state["batch"]
        b.run(state["dt"], state["steps"])
        got = [b.get_energies(k) for k in range(len(state["arrays"]))]
        return {"e": np.concatenate([g[0] for g in got]), "E": np.concatenate([g[1] for g in got])}
    if state["kind"] == "serve":
        srv = state["server"]
        ids = [srv.submit(c, a, a.e, a.E, state["steps"], state["dt"])
               for c, a in zip(state["cfgs"], state["arrays"])]
        for i in ids:
            srv.wait(i)
        got = [srv.result(i) for i in ids]
        return {"e": np.concatenate([g[0] for g in got]), "E": np.concatenate([g[1] for g in got])}
    S, L = state["solver"], state["lattice"]
    arrays = [state[k] for k in ("mass", "rho", "h", "sigma0")] + [L["kind"], L["copy_of"],
                                                                  state["e"], state["E"]]
    S.set_particles_device(L["pos"].shape[0], _ptr(L["pos"]), *[_ptr(a) for a in arrays])
    if state["kind"] == "moving":
        S.adapt_smoothing_lengths(eta=4.0)
    for k, ins in enumerate(state["inputs"]):
        if k and state["moves"]:
            S.move_particles_device(_ptr(state["moves"][k - 1]))
        S.step_device(state["dt"], *[_ptr(t) for t in ins])
    S.get_energies_device(_ptr(state["e_out"]), _ptr(state["E_out"]))
    return {"e": state["e_out"], "E": state["E_out"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without: every input read once and every result written
# once; per neighbour pair the geometry (~20 operations) once per particle set
# and, per step, its operator value (3) and one product in each of two outer
# iterations (4)
# ---------------------------------------------------------------------------
def work(case):
    if case["kind"] in ("batch", "serve"):
        # mean of a log-uniform size
        lo, hi = case["nmin"], case["nmax"]
        mean = (hi - lo) / math.log(hi / lo) if hi > lo else lo
        n, pairs = case["count"] * mean, 24 if case.get("dim", 3) == 2 else 92
        dim, sets, fields = case.get("dim", 3), 1, 0
    else:
        counts = [c for c in (case["nx"], case["ny"], case["nz"]) if c]
        dim = len(counts)
        wide = case.get("problem") == "cgs" or case["kind"] == "moving"
        if case.get("problem") == "cgs":
            counts = [counts[0]] * dim
        n = math.prod(counts)
        pairs = {2: 44 if wide else 24, 3: 250 if wide else 101}[dim]
        sets = case["steps"] + 1 if case["kind"] == "moving" else 1
        fields = 4 if case.get("problem", "mms") in ("mms", "mms-lp", "cgs") else 0
    per = 8 * dim + 60 + 16 + 8 * fields * case["steps"] + 8 * dim * (sets - 1)
    return {"bytes": float(per * n),
            "flops": float(n * pairs * (20 * sets + 7 * case["steps"]))}


# ---------------------------------------------------------------------------
# the same equations in 64-bit torch
# ---------------------------------------------------------------------------
def _dw(kern, dim, r, h):
    """dW/dr of the cubic B-spline (support 2h) or the Wendland C4 kernel (support h)."""
    q = r / h
    if kern == WENDLAND:
        k = {1: 1.5, 2: 36.0 / (5.0 * math.pi), 3: 45.0 / (4.0 * math.pi)}[dim]
        w = torch.where(q <= 1.0, -14.0 * q * (1.0 + 4.0 * q) * (1.0 - q) ** 4, 0.0)
    else:
        k = {1: 2.0 / 3.0, 2: 10.0 / (7.0 * math.pi), 3: 1.0 / math.pi}[dim]
        w = torch.where(q < 1.0, -3.0 * q + 2.25 * q * q,
                        torch.where(q < 2.0, -0.75 * (2.0 - q) ** 2, 0.0))
    return k * w / h ** (dim + 1)


def _offsets(p, reach):
    """(row, column) of the lattice offsets within `reach` spacings of every interior point."""
    L = p["lattice"]
    dim, ext = L["dim"], L["ext"]
    rows = torch.nonzero(L["kind"] == INTERIOR).flatten()
    idx, lin = [], rows.clone()
    for d in range(dim):
        idx.append(lin % ext[d])
        lin = lin // ext[d]
    span = range(-reach, reach + 1)
    for off in np.stack(np.meshgrid(*[span] * dim, indexing="ij"), -1).reshape(-1, dim).tolist():
        if not any(off) or sum(max(0, abs(o) - 0.3) ** 2 for o in off) > (reach + 0.3) ** 2:
            continue
        ok = torch.ones_like(rows, dtype=torch.bool)
        shift, stride = 0, 1
        for d in range(dim):
            ok &= (idx[d] + off[d] >= 0) & (idx[d] + off[d] < ext[d])
            shift += off[d] * stride
            stride *= ext[d]
        yield rows[ok], rows[ok] + shift


def _pairs(p):
    """Neighbour pairs r < s max(h_i, h_j) of the interior rows: i, j, F_ij, x_i - x_j."""
    kern, dim = p["phys"]["kernel"], p["phys"]["dim"]
    s = 1.0 if kern == WENDLAND else 2.0
    x, h = p["lattice"]["pos"], p["h"]
    reach = int(math.floor(s * float(h.max()) / p["lattice"]["dx"] + 2.0 * p["lattice"]["jitter"]))
    parts = []
    for i, j in _offsets(p, reach):
        r2 = ((x[i] - x[j]) ** 2).sum(1)
        m = r2 < (s * torch.maximum(h[i], h[j])) ** 2
        parts.append((i[m], j[m]))
    i, j = torch.cat([a for a, _ in parts]), torch.cat([b for _, b in parts])
    order = torch.argsort(i, stable=True)
    i, j = i[order], j[order]
    d = x[i] - x[j]
    r = d.norm(dim=1)
    return i, j, 0.5 * (_dw(kern, dim, r, h[i]) + _dw(kern, dim, r, h[j])) / r, d


def _density(kern, dim, r, h):
    q = r / h
    if kern == WENDLAND:
        k = {1: 1.5, 2: 36.0 / (5.0 * math.pi), 3: 45.0 / (4.0 * math.pi)}[dim]
        w = torch.where(q <= 1.0, (1.0 - q) ** 5 * (8.0 * q * q + 5.0 * q + 1.0), 0.0)
    else:
        k = {1: 2.0 / 3.0, 2: 10.0 / (7.0 * math.pi), 3: 1.0 / math.pi}[dim]
        w = torch.where(q < 1.0, 1.0 - 1.5 * q * q + 0.75 * q ** 3,
                        torch.where(q < 2.0, 0.25 * (2.0 - q) ** 3, 0.0))
    return k * w / h ** dim


def _adapted(p, eta):
    """Smoothing lengths of the initialisation iteration, to rounding."""
    kern, dim = p["phys"]["kernel"], p["phys"]["dim"]
    s = 1.0 if kern == WENDLAND else 2.0
    x, h, kind = p["lattice"]["pos"], p["h"].clone(), p["lattice"]["kind"]
    found = [(i, (x[i] - x[j]).norm(dim=1)) for i, j in _offsets(p, p["lattice"]["layers"] + 1)]
    i, r = torch.cat([a for a, _ in found]), torch.cat([b for _, b in found])
    inner = kind == INTERIOR
    for _ in range(100):
        S = _density(kern, dim, torch.zeros_like(h), h)
        S.index_add_(0, i, _density(kern, dim, r, h[i]))
        new = h * (eta / s) / (h ** dim * S) ** (1.0 / dim)
        new = torch.where(inner, torch.minimum(torch.maximum(new, 0.5 * h), 2.0 * h), h)
        done = bool(((new - h).abs() <= 1e-13 * new).all())
        h = new
        if done:
            break
    return h


def _cg(A, diag, V, b, x):
    """Jacobi-preconditioned CG on V A x = V b, to rounding."""
    def mul(v):
        return diag * v + torch.mv(A, v)

    r = b - mul(x)
    stop, best, stale = 1e-15 * b.norm(), math.inf, 0
    pd, rho = torch.zeros_like(b), None
    for _ in range(2000):
        rn = float(r.norm())
        best, stale = (rn, 0) if rn < 0.9 * best else (best, stale + 1)
        if rn <= stop or stale > 6:
            break
        z = r / diag
        rho_new = torch.dot(V * r, z)
        pd = z if rho is None else z + (rho_new / rho) * pd
        rho = rho_new
        q = mul(pd)
        alpha = rho / torch.dot(V * pd, q)
        x = x + alpha * pd
        r = r - alpha * q
    return x


def _geometry(p):
    i, j, F, d = _pairs(p)
    L = p["lattice"]
    src = torch.where(L["kind"] == COPY, L["copy_of"], torch.arange(len(L["kind"]), device=i.device))
    return dict(i=i, j=j, js=src[j], F=F, d=d, src=src)


def _advance(p, G, e, E, ins):
    """One backward-Euler step with nonlinear elimination, every loop to rounding."""
    ph, dt, kind = p["phys"], p["dt"], p["lattice"]["kind"]
    i, j, js, F, src = G["i"], G["j"], G["js"], G["F"], G["src"]
    n, V, rho = e.numel(), p["mass"] / p["rho"], p["rho"]
    inner = kind == INTERIOR
    rows = torch.nonzero(inner).flatten()
    a, c, cv = ph["a"], ph["c"], ph["cv"]
    T = e / cv
    sig = p["sigma0"] * T ** ph["opacity_exp"] if ph["opacity_exp"] else p["sigma0"].clone()
    f = 1.0 / (1.0 + c * sig * dt * 4.0 * a * T ** 3 / (rho * cv))
    R = torch.zeros_like(e)
    if ph["limiter"]:
        g = torch.zeros(n, ph["dim"], dtype=F64, device=e.device)
        g.index_add_(0, i, (V[j] * (E[js] - E[i]) * F)[:, None] * G["d"])
        R = torch.where(inner, g.norm(dim=1) / ((sig + ph["sigma_s"]) * E), R)
    D = c * _limiter(R, ph["limiter"])[0] / (sig + ph["sigma_s"])
    D, f, sig = D[src], f[src], sig[src]
    Qe, QE, ge, gE = ins
    ghost = kind == DIRICHLET
    if gE is not None:
        E = torch.where(ghost, gE, E)
    w = -V[j] * (D[i] + D[j]) * F
    diag = (1.0 / dt + c * sig * f).index_add(0, i, w)[rows]
    fixed = ghost[j]
    gb = torch.zeros_like(e).index_add_(0, i[fixed], w[fixed] * E[j[fixed]])[rows]
    place = torch.full((n,), -1, dtype=torch.int64, device=e.device)
    place[rows] = torch.arange(len(rows), device=e.device)
    m = ~fixed
    ptr = torch.zeros(len(rows) + 1, dtype=torch.int64, device=e.device)
    ptr[1:] = torch.cumsum(torch.bincount(place[i[m]], minlength=len(rows)), 0)
    A = torch.sparse_csr_tensor(ptr, place[js[m]], -w[m], size=(len(rows), len(rows)))
    Vi, si, fi, ri = V[rows], sig[rows], f[rows], rho[rows]
    e0, E0 = e[rows], E[rows]
    qe = 0.0 if Qe is None else Qe[rows]
    qE = 0.0 if QE is None else QE[rows]

    def material(Enew, start):
        v, P = start, c * si * Enew + qe
        for _ in range(50):
            t = v / cv
            de = (ri / dt * (v - e0) + c * si * a * t ** 4 - P) / (ri / dt + 4 * c * si * a * t ** 3 / cv)
            v = v - de
            if bool((de.abs() <= 1e-15 * v.abs()).all()):
                break
        return v

    el, El, last = material(E0, e0), E0, math.inf
    for _ in range(200):
        b = E0 / dt + c * si * a * (el / cv) ** 4 - (1.0 - fi) * c * si * El + qE + gb
        Enew = _cg(A, diag, Vi, b, El)
        enew = material(Enew, el)
        change = max(float(((Enew - El) / Enew).abs().max()), float(((enew - el) / enew).abs().max()))
        el, El = enew, Enew
        if change < 1e-14 or (change < 1e-11 and change > 0.5 * last):
            break
        last = change
    e, E = e.clone(), E.clone()
    if ge is not None:
        e = torch.where(ghost, ge, e)
    e[rows], E[rows] = el, El
    return e[src], E[src]


def _joined(problems):
    """Independent problems of one physics as one: their pairs and arrays end to end."""
    at, parts = 0, []
    for q in problems:
        G = _geometry(q)
        parts.append({k: (v if k in ("F", "d") else v + at) for k, v in G.items()})
        at += q["e"].numel()
    G = {k: torch.cat([g[k] for g in parts]) for k in parts[0]}
    p = {k: torch.cat([q[k] for q in problems]) for k in ("mass", "rho", "sigma0", "e", "E")}
    p.update(phys=problems[0]["phys"], dt=problems[0]["dt"],
             lattice=dict(kind=torch.cat([q["lattice"]["kind"] for q in problems])))
    return p, G


def _to(p, dev):
    q = {k: (v.to(dev) if torch.is_tensor(v) else v) for k, v in p.items()}
    q["lattice"] = {k: (v.to(dev) if torch.is_tensor(v) else v) for k, v in p["lattice"].items()}
    return q


def exact(case, seed):
    dev = torch.device("cuda")
    none = (None, None, None, None)
    if case["kind"] in ("batch", "serve"):
        problems = [_to(p, dev) for p in _small_waves(case, seed, "cpu")]
        got = [None] * len(problems)
        for dim in (2, 3):
            mine = [k for k, p in enumerate(problems) if p["phys"]["dim"] == dim]
            if not mine:
                continue
            p, G = _joined([problems[k] for k in mine])
            e, E = p["e"], p["E"]
            for _ in range(case["steps"]):
                e, E = _advance(p, G, e, E, none)
            at = 0
            for k in mine:
                n = problems[k]["e"].numel()
                got[k] = (e[at:at + n], E[at:at + n])
                at += n
        return {"e": torch.cat([g[0] for g in got]).cpu().numpy(),
                "E": torch.cat([g[1] for g in got]).cpu().numpy()}
    p = _problem(case, seed, dev)
    if case["kind"] == "moving":
        p["h"] = _adapted(p, 4.0)
    e, E = p["e"], p["E"]
    # copy ghosts hold their particle's energies once a step is done; before the
    # first one only the particle's own values are read
    G = _geometry(p)
    for k, ins in enumerate(p["inputs"]):
        if k and p["moves"]:
            p["lattice"]["pos"] = p["moves"][k - 1]
            G = _geometry(p)
        e, E = _advance(p, G, e, E, ins)
    return {"e": e, "E": E}
