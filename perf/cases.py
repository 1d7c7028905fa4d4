"""The work that users have this solver do, as measurable cases.

Kinds of case, each through the package's public entry points:
  solve   one-shot solves of small problems, stopped by a per-step rule: the
          paper's 1D experiments and the 2D sinusoid
  plan    a device-resident plan: load a source, advance a number of sweeps
          with residual checks, read the potential (a 3D solve's steady part)
  ladder  one-shot solves from host buffers with a precision ladder
  batch   many uneven 3D grids in one context, driven by the caller
  serve   requests with mixed tolerances from host buffers, in a context whose
          own thread drives them
  fft     the scheme's exact fixed point by FFT

Sources are the solver's workloads: periodic Gaussians of alternating charge
(stiff) and products of sinusoids (smooth).
"""
import math

import torch

import paper_1504_05869_gb300 as pk

CHECK = 32    # steps between residual checks, as the benchmark uses


def listed():
    return [
        # the paper's Table 2: 1D, order 7, tau_lb = 1, thousands of tiny steps (the smallest calls)
        dict(name="solve_1d_L64", kind="solve", lattice="D1Q13", order=7, nx=64, ny=1, nz=1,
             tau=1.0, kn=0.0, tol=1e-13, tol_kind="rel_l2"),
        # the 2D sinusoid on the two-dimensional high-order set, stopped at max|dPhi| per sweep
        dict(name="solve_2d_64_kn0.1", kind="solve", lattice="D2Q169", order=7, nx=64, ny=64, nz=1,
             tau=0.0, kn=0.1, tol=1e-12, tol_kind="max_abs"),
        # the benchmark's line: 256^3, binary64-accurate fixed-point storage
        dict(name="plan_fx64_256", kind="plan", lattice="D3Q111", order=5, precision="fx64",
             nx=256, ny=256, nz=256, tau=0.0, kn=0.2, steps=32),
        # binary64 storage on a ragged grid (rows that are no whole tiles)
        dict(name="plan_fp64_173x141x100", kind="plan", lattice="D3Q111", order=5, precision="fp64",
             nx=173, ny=141, nz=100, tau=0.0, kn=0.2, steps=32),
        # binary32 storage, the first rung of mixed-precision solves
        dict(name="plan_fp32_192", kind="plan", lattice="D3Q111", order=5, precision="fp32",
             nx=192, ny=192, nz=192, tau=0.0, kn=0.2, steps=32),
        # binary16 storage, the first rung of the three-step ladder
        dict(name="plan_fp16_256", kind="plan", lattice="D3Q111", order=5, precision="fp16",
             nx=256, ny=256, nz=256, tau=0.0, kn=0.2, steps=32),
        # standard first-order lattice Boltzmann, the comparison every solve is held against
        dict(name="plan_d3q19_fp64_256", kind="plan", lattice="D3Q19", order=1, precision="fp64",
             nx=256, ny=256, nz=256, tau=0.0, kn=0.2, steps=32),
        # tau_lb = 1, the paper's own setting in 3D (scalar steps)
        dict(name="plan_tau1_256", kind="plan", lattice="D3Q111", order=5, precision="fp64",
             nx=256, ny=256, nz=256, tau=1.0, kn=0.0, steps=32),
        # a mid-size 3D solve from host arrays: binary32 steps, then 64-bit fixed point
        dict(name="ladder_fx64_80x48x64", kind="ladder", lattice="D3Q111", order=5,
             precision="mixed_fx64", nx=80, ny=48, nz=64, tau=0.0, kn=0.2, tol=1e-10),
        # independent uneven grids advanced together (parameter studies)
        dict(name="batch_fp32_16", kind="batch", lattice="D3Q111", order=5, precision="fp32",
             count=16, lo=32, hi=128, kn=0.2, tol=1e-6, pick=2),
        # a served burst: mixed tolerances, host buffers, binary32 then binary64
        dict(name="serve_mixed_6", kind="serve", lattice="D3Q111", order=5, precision="mixed",
             count=6, lo=32, hi=112, kn=0.2, tol=1e-10, pick=3),
        # the direct comparator on a mid-size grid of no special sizes
        dict(name="fft_200x180x150", kind="fft", lattice="D3Q111", order=5, nx=200, ny=180, nz=150,
             tau=0.0, kn=0.2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi, most):
    """Three edges in [lo, hi] with at most `most` sites; x whole 64-site tiles half of the time."""
    while True:
        n = [_log_int(rng, lo, hi) for _ in range(3)]
        if rng.random() < 0.5:
            n[0] = max(64, 64 * (n[0] // 64))
        if n[0] * n[1] * n[2] <= most:
            return n


def draw(rng):
    kind = rng.choice(["solve", "solve", "plan", "plan", "plan", "ladder", "batch", "serve", "fft"])
    if kind == "solve":
        if rng.random() < 0.5:
            lat, order, hi = rng.choice([("D1Q5", 1, 72), ("D1Q5", 3, 72), ("D1Q9", 5, 100),
                                         ("D1Q13", 7, 128)])
            return dict(kind=kind, lattice=lat, order=order, nx=_log_int(rng, 16, hi), ny=1, nz=1,
                        tau=1.0, kn=0.0, tol=rng.choice([1e-11, 1e-12, 1e-13]), tol_kind="rel_l2")
        lat, order, hi = rng.choice([("D2Q25", 3, 56), ("D2Q81", 5, 72), ("D2Q169", 7, 80)])
        paper = rng.random() < 0.5
        return dict(kind=kind, lattice=lat, order=order, nx=_log_int(rng, 24, hi),
                    ny=_log_int(rng, 24, hi), nz=1, tau=1.0 if paper else 0.0,
                    kn=0.0 if paper else rng.choice([0.1, 0.2]), tol=1e-12, tol_kind="max_abs")
    if kind == "plan":
        lat, order = rng.choice([("D3Q111", 5), ("D3Q111", 5), ("D3Q111", 5), ("D3Q19", 1)])
        prec = rng.choice(["fx64", "fp64", "fp32", "fp16", "tau1"])
        nx, ny, nz = _box(rng, 40, 256, 1 << 24)
        tau1 = prec == "tau1"
        return dict(kind=kind, lattice=lat, order=order, precision="fp64" if tau1 else prec,
                    nx=nx, ny=ny, nz=nz, tau=1.0 if tau1 else 0.0,
                    kn=0.0 if tau1 else rng.choice([0.05, 0.2, 0.5]), steps=rng.choice([16, 24, 32]))
    if kind == "ladder":
        nx, ny, nz = _box(rng, 24, 96, 300000)
        return dict(kind=kind, lattice="D3Q111", order=5,
                    precision=rng.choice(["mixed", "mixed_fx64", "fx64", "fp64"]), nx=nx, ny=ny,
                    nz=nz, tau=0.0, kn=0.2, tol=rng.choice([1e-8, 1e-10]))
    if kind == "batch":
        return dict(kind=kind, lattice="D3Q111", order=5,
                    precision=rng.choice(["fp32", "fp32", "fp64", "fx64"]),
                    count=rng.randint(4, 12), lo=32, hi=rng.choice([64, 96]), kn=0.2, tol=1e-6,
                    pick=rng.randint(4, 1000))
    if kind == "serve":
        return dict(kind=kind, lattice="D3Q111", order=5,
                    precision=rng.choice(["mixed", "mixed_fx64"]), count=rng.randint(2, 6), lo=32,
                    hi=rng.choice([64, 88]), kn=0.2, tol=1e-10, pick=rng.randint(4, 1000))
    lat, order = rng.choice([("D3Q111", 5), ("D3Q111", 5), ("D3Q19", 1)])
    nx, ny, nz = _box(rng, 40, 256, 1 << 23)
    return dict(kind="fft", lattice=lat, order=order, nx=nx, ny=ny, nz=nz, tau=0.0,
                kn=rng.choice([0.05, 0.2]))


# ---------------------------------------------------------------- inputs

def _shape(c):
    """numpy order, as many axes as the lattice has."""
    dim = int(c["lattice"][1])
    return (c["nz"], c["ny"], c["nx"])[3 - dim:]


def _sinusoid(shape, g):
    """A product of sinusoids, one period per axis, at a random phase."""
    out = torch.ones((), dtype=torch.float64, device="cuda")
    for n in shape:
        ph = 2 * math.pi * float(torch.rand((), generator=g, dtype=torch.float64))
        x = torch.arange(n, dtype=torch.float64, device="cuda")
        out = out[..., None] * torch.sin(2 * math.pi * x / n + ph)
    return out


def _gaussians(shape, count, sig_lo, sig_hi, g):
    """`count` periodic 3D Gaussians, charges alternating +1, -1, centres and widths random."""
    u = torch.rand((count, 4), generator=g, dtype=torch.float64)
    sig = sig_lo + (sig_hi - sig_lo) * u[:, 3]
    q = torch.tensor([1.0 - 2.0 * (j % 2) for j in range(count)], dtype=torch.float64)
    ax = []
    for a, n in enumerate(shape):
        d = (torch.arange(n, dtype=torch.float64)[None] - n * u[:, a:a + 1]).abs()
        d = torch.minimum(d, n - d)
        ax.append(torch.exp(-d * d / (2 * sig[:, None] ** 2)))
    ax[0] = ax[0] * (q * (2 * math.pi * sig * sig) ** -1.5)[:, None]
    ax = [a.cuda() for a in ax]
    zy = (ax[0][:, :, None] * ax[1][:, None, :]).reshape(count, -1)
    return (zy.t() @ ax[2]).reshape(shape).contiguous()


def _jobs(c):
    """Shapes and tolerances of a batch or a burst: what the case stands for, whatever the seed."""
    g = torch.Generator().manual_seed(1000 + c["pick"])
    jobs = []
    for j in range(c["count"]):
        u = torch.rand(4, generator=g, dtype=torch.float64).tolist()
        n = [int(round(math.exp(math.log(c["lo"]) + v * math.log(c["hi"] / c["lo"])))) for v in u[:3]]
        jobs.append((tuple(n), 1 + int(16 * u[3])))
    return jobs


def _sources(c, seed):
    """The source arrays of a case, on the GPU."""
    g = torch.Generator().manual_seed(int(seed))
    if c["kind"] in ("batch", "serve"):
        return [_gaussians(shape, k, 1.0, 4.0, g) if c["kind"] == "batch" or j % 2 == 0
                else _sinusoid(shape, g) for j, (shape, k) in enumerate(_jobs(c))]
    if c["kind"] == "solve":
        return [_sinusoid(_shape(c), g)]
    return [_gaussians(_shape(c), 64 if c["kind"] == "plan" else 16, 2.0, 2.0, g)]


def _tol(c, j):
    """Tolerance of request j: a batch's own, a burst's in turn."""
    return c["tol"] if c["kind"] != "serve" else (1e-6, 1e-8, 1e-10)[j % 3]


def _problem(c, **kw):
    return pk.problem(c["lattice"], _shape(c), c["order"], tau_lb=c["tau"], knudsen=c["kn"], **kw)


def prepare(case, seed):
    c = dict(case)
    rho = _sources(c, seed)
    kind = c["kind"]
    if kind == "plan":
        plan = pk.Plan(_problem(c, precision=c["precision"], check_every=CHECK, max_sweeps=1 << 20))
        return dict(c=c, rho=rho[0], phi=torch.empty_like(rho[0]), plan=plan)
    if kind in ("solve", "fft"):
        prob = _problem(c, tol=c.get("tol", 0.0), tol_kind=c.get("tol_kind", "rel_l2"),
                        check_every=1, max_sweeps=1 << 20)
        return dict(c=c, rho=rho[0], phi=torch.empty_like(rho[0]), prob=prob)
    if kind == "ladder":
        r = rho[0].cpu()
        prob = _problem(c, tol=c["tol"], precision=c["precision"], check_every=CHECK,
                        max_sweeps=1 << 20)
        return dict(c=c, rho=r, phi=torch.empty_like(r), prob=prob)
    if kind == "serve":
        rho = [r.cpu() for r in rho]
    ctx = pk.Context(c["lattice"], c["order"], precision=c["precision"], check_every=CHECK,
                     hbm_budget_bytes=60 * 10 ** 9, threaded=kind == "serve")
    return dict(c=c, rho=rho, phi=[torch.empty_like(r) for r in rho], ctx=ctx)


def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind == "plan":
        plan = state["plan"]
        plan.load_source(state["rho"])
        plan.run(c["steps"], check_every=CHECK)
        return plan.phi(state["phi"])
    if kind in ("solve", "ladder"):
        pk.solve(state["rho"], state["phi"], state["prob"])
        return state["phi"]
    if kind == "fft":
        pk.fixed_point_fft(state["rho"], state["phi"], state["prob"])
        return state["phi"]
    ctx = state["ctx"]
    tickets = [ctx.submit(r, p, knudsen=c["kn"], tol=_tol(c, j), max_sweeps=1 << 20)
               for j, (r, p) in enumerate(zip(state["rho"], state["phi"]))]
    if kind == "batch":
        ctx.run()
    for t in tickets:
        ctx.wait(t)
        ctx.release(t)
    return state["phi"]


# ---------------------------------------------------------------- work

_Q = {"D1Q5": 5, "D1Q9": 9, "D1Q13": 13, "D2Q25": 25, "D2Q81": 81, "D2Q169": 169, "D3Q19": 19,
      "D3Q111": 111}
_BYTES = {"fp64": 8, "fx64": 8, "fp32": 4, "fp16": 2}


def work(case):
    """The source read once, the potential written once, and, where the populations are larger
    than the chip holds, each read and written once per step.  A step costs three operations per
    population (its share of the density, one multiply-add), a scalar step two."""
    c = dict(case)
    Q = _Q[c["lattice"]]
    if c["kind"] in ("batch", "serve"):
        sites = [s[0] * s[1] * s[2] for s, _ in _jobs(c)]
        e = _BYTES.get(c["precision"], 4)
        # residual per step falls by about a tenth of a decade in 5 steps at this Knudsen number
        steps = [60 * -math.log10(_tol(c, j)) / 2 for j in range(len(sites))]
        upd = sum(v * n for v, n in zip(sites, steps))
        return {"bytes": 16.0 * sum(sites) + upd * (2 * Q * e + e), "flops": 3.0 * Q * upd}
    V = c["nx"] * c["ny"] * c["nz"]
    if c["kind"] == "fft":
        # forward and inverse real transforms, and the transfer function of half the spectrum
        return {"bytes": 16.0 * V, "flops": 5.0 * V * math.log2(V) + V / 2 * 10.0 * Q}
    if c["kind"] == "plan":
        n = c["steps"] + 1
        if c["tau"] == 1.0:
            return {"bytes": 16.0 * V + n * V * 24.0, "flops": 2.0 * Q * V * n}
        e = _BYTES[c["precision"]]
        return {"bytes": 16.0 * V + n * V * (2.0 * Q * e + max(e, 4)), "flops": 3.0 * Q * V * n}
    if c["kind"] == "ladder":
        n = 30 * -math.log10(c["tol"])
        e = _BYTES.get(c["precision"], 4)
        return {"bytes": 16.0 * V + n * V * (2.0 * Q * e + e), "flops": 3.0 * Q * V * n}
    # solves whose state fits on the chip: steps grow with the square of the longest edge at tau 1
    n = 210 if c["tau"] == 0.0 else 0.25 * max(c["nx"], c["ny"]) ** 2
    return {"bytes": 16.0 * V, "flops": (3.0 if c["tau"] == 0.0 else 2.0) * Q * V * n}


# ---------------------------------------------------------------- exact values

# Speeds and weights of the velocity sets (the paper's Appendix; D3Q111 by shell), and c_s^2.
_SETS = {
    5: (0.3675444679663241, {0: 0.6366469031260782, 1: 0.18141458774368577,
                             3: 0.0002619606932751435}),
    9: (0.7560808525942686, {0: 0.4581351555076766, 1: 0.23734280857794043,
                             2: 0.032324653788654935, 3: 0.001264062151536515,
                             5: 8.977280298192933e-07}),
    13: (1.3326518154047418, {0: 0.3455934552621565, 1: 0.2374599218260301, 2: 0.0770573099396458,
                              3: 0.011801423732312036, 4: 0.0008552466009513439,
                              5: 2.884934614927074e-05, 6: 5.209238332209471e-07}),
}
_SHELLS = {
    "D3Q19": (1 / 3, {(0, 0, 0): 1 / 3, (1, 0, 0): 1 / 18, (1, 1, 0): 1 / 36}),
    "D3Q111": (0.6979533220196831, {
        (0, 0, 0): 0.15014405211326798, (1, 0, 0): 0.02500398840704123,
        (1, 1, 0): 0.04505812049781918, (2, 0, 0): 0.010549030462576969,
        (2, 1, 1): 0.0034941797555202033, (2, 2, 0): 0.0006031099650419177,
        (3, 0, 0): 4.500168524455985e-05, (3, 1, 0): 0.00018120734608628378,
        (3, 3, 0): 9.792909088441143e-06, (3, 3, 3): 7.817069506635642e-07}),
}


def _lattice(name, order):
    """Velocities (x, y, z), equilibrium and source weights (Hermite forms of the order), c_s^2."""
    dim, Q = int(name[1]), int(name[3:])
    vel, w = [], []
    if dim == 3:
        cs2, shells = _SHELLS[name]
        r = range(-3, 4)
        for v in ((x, y, z) for z in r for y in r for x in r):
            key = tuple(sorted((abs(a) for a in v), reverse=True))
            if key in shells:
                vel.append(v)
                w.append(shells[key])
    else:
        cs2, line = _SETS[round(Q ** (1 / dim))]
        one = [(s * v, wt) for v, wt in line.items() for s in ((1, -1) if v else (1,))]
        for x, wx in one:
            for y, wy in (one if dim == 2 else [(0, 1.0)]):
                vel.append((x, y, 0))
                w.append(wx * wy)
    assert len(vel) == Q
    D, phi, chi = dim, [], []
    for v, wt in zip(vel, w):
        x2 = sum(a * a for a in v) / cs2
        H2 = x2 - D
        H4 = x2 ** 2 - 2 * (D + 2) * x2 + D * (D + 2)
        H6 = x2 ** 3 - 3 * (D + 4) * x2 ** 2 + 3 * (D + 2) * (D + 4) * x2 - D * (D + 2) * (D + 4)
        phi.append(wt * (1.0 - (H4 / 8 if order >= 5 else 0) + (H6 / 24 if order >= 7 else 0)))
        chi.append(wt * (1.0 - (H2 / 2 if order >= 3 else 0) + (H4 / 8 if order >= 5 else 0)
                         - (H6 / 48 if order >= 7 else 0)))
    t = dict(dtype=torch.float64, device="cuda")
    return vel, torch.tensor(phi, **t), torch.tensor(chi, **t), cs2


def _evolve(rho, lat, order, tau, kn, steps=None, tol=0.0, kind="rel_l2", first=0, every=1):
    """Phi after `steps` steps, or at the first check (steps first, first + every, ...) whose
    change of Phi is below tol."""
    vel, phi, chi, cs2 = _lattice(lat, order)
    shape = rho.shape
    if tau <= 0:
        tau = 0.5 + kn * min(n for n in shape if n > 1) / math.sqrt(cs2)
    om = 1.0 / tau
    S = ((rho - rho.mean()) * (cs2 * (tau - 0.5))).reshape(1, -1)
    V = S.numel()
    sites = torch.arange(V, device="cuda").reshape(shape)
    axes = [2 - a for a in range(3 - len(shape), 3)]       # component of each array axis
    idx = torch.empty((len(vel), V), dtype=torch.int64, device="cuda")
    for i, v in enumerate(vel):
        idx[i] = torch.roll(sites, [v[k] for k in axes], list(range(len(shape)))).reshape(-1) + i * V
    f = torch.zeros((len(vel), V), dtype=torch.float64, device="cuda")
    g = torch.empty_like(f)
    wphi, chi = (om * phi)[:, None], chi[:, None]
    old, k = None, 0
    while True:
        torch.take(f, idx, out=g)
        Phi = g.sum(0, keepdim=True)
        if steps is not None and k == steps:
            return Phi.reshape(shape)
        if steps is None and k >= max(1, first) and (k - first) % every == 0:
            d = Phi - old
            r = d.abs().max() if kind == "max_abs" else d.norm() / Phi.norm()
            if float(r) < tol:
                return Phi.reshape(shape)
        g.mul_(1.0 - om).addcmul_(wphi, Phi).addcmul_(chi, S)
        f, g, old, k = g, f, Phi, k + 1


def _fixed_point(rho, lat, order, tau, kn):
    vel, phi, chi, cs2 = _lattice(lat, order)
    shape = rho.shape
    if tau <= 0:
        tau = 0.5 + kn * min(n for n in shape if n > 1) / math.sqrt(cs2)
    a = 1.0 - 1.0 / tau
    S = torch.fft.rfftn((rho - rho.mean()) * (cs2 * (tau - 0.5)))
    ks = [2 * math.pi * torch.arange(S.shape[d], dtype=torch.float64, device="cuda") / n
          for d, n in enumerate(shape)]
    num, den = torch.zeros_like(S.real), torch.zeros_like(S.real)
    for v, p, x in zip(vel, phi.tolist(), chi.tolist()):
        th = v[2] * ks[0][:, None, None] + v[1] * ks[1][None, :, None] + v[0] * ks[2][None, None, :]
        c, s, o = th.cos(), th.sin(), 2 * (th / 2).sin() ** 2      # e = c - i s, o = 1 - c
        dr, di = 1.0 - a * c, a * s
        m = dr * dr + di * di
        num += x * (c * dr - s * di) / m
        den += p * (o * dr + s * di) / m
    num[0, 0, 0], den[0, 0, 0] = 0.0, 1.0
    return torch.fft.irfftn(S * (num / den), s=shape)


def exact(case, seed):
    c = dict(case)
    rho = _sources(c, seed)
    if c["kind"] in ("batch", "serve"):
        # a request's checks come at steps CHECK - 1, 2 CHECK - 1, ...
        return [_evolve(r, c["lattice"], c["order"], 0.0, c["kn"], tol=_tol(c, j), first=CHECK - 1,
                        every=CHECK).to("cuda" if c["kind"] == "batch" else "cpu")
                for j, r in enumerate(rho)]
    args = (rho[0], c["lattice"], c["order"], c["tau"], c["kn"])
    if c["kind"] == "fft":
        return _fixed_point(*args)
    if c["kind"] == "plan":
        return _evolve(*args, steps=c["steps"])
    if c["kind"] == "ladder":
        return _evolve(*args, tol=c["tol"], first=CHECK, every=CHECK).cpu()
    return _evolve(*args, tol=c["tol"], kind=c["tol_kind"], first=1)
