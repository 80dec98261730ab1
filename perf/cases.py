"""The work that users of the framework have it do, as timed cases through its public entry points.

Lattices, couplings and fields follow the repository's configurations: L x L x Nt from 4 x 4 x 8 (the
dense cross-check) over 20 x 20 x 40 and 40 x 40 x 80 (single chains), 64 uneven chains in one batch, to
80 x 80 x 160 with eight right-hand sides (the benchmark). A pass is one call that a program makes in its
loop: an operator application, a solve, an action with its gradient, a drift, a trajectory. Boson fields
are ordered states (the mean-field amplitude of the right-hand side count on one component, plus
free-boson fluctuations), as a thermalised chain has them; the smallest lattice starts from N(0, 1).

Solves run to a true residual of 1e-12: there the solution, the force and the new field are settled to
about ten digits whatever order a solver adds its terms in (at 1e-10 the stopping point shows).

``exact`` gives the same quantities in 64 bits from plain torch, written from the model's definition.
"""

import math

import torch

from paper_2204_14241_gb300 import hmc, presets
from paper_2204_14241_gb300.action import pseudofermion_action

MODEL = presets.baseline()
TOL = 1e-12
NOMINAL_ITERATIONS = 100   # CG steps that a solve's arithmetic is counted with (work); real counts are 90 to 500

# even extents and slice counts the FFTs take (factors 2, 3, 5, 7)
EXTENTS = [n for n in range(4, 81, 2) if all(p <= 7 for p in range(2, n + 1)
                                            if n % p == 0 and all(p % q for q in range(2, p)))]
SLICES = [n for n in range(4, 161) if all(p <= 7 for p in range(2, n + 1)
                                         if n % p == 0 and all(p % q for q in range(2, p)))]


def listed():
    return [
        # the smallest call: one update of the dense-cross-check chain, FP64; launches and latency are all it costs
        dict(name="trajectory_4_fp64", kind="trajectory", L=4, Nt=8, nrhs=1, solver="fp64", precond=True, guess=0,
             n_leap=10, field="normal"),
        # one solve of the 20 x 20 x 40 chain with the defaults (mixed precision, preconditioned), as a force or
        # a measurement asks for it
        dict(name="solve_20_pcg", kind="solve", L=20, Nt=40, nrhs=1, solver="mixed", precond=True),
        # an extent and a slice count no table is made for, an odd number of right-hand sides, plain CG
        dict(name="solve_18_odd", kind="solve", L=18, Nt=35, nrhs=3, solver="mixed", precond=False),
        # the plain FP64 solver at the size of the largest batched chain
        dict(name="solve_24_fp64", kind="solve", L=24, Nt=48, nrhs=2, solver="fp64", precond=False),
        # the fermionic observable: eight +-1 probes through the twisted Fourier basis, one multi-RHS solve
        dict(name="green_16", kind="green", L=16, Nt=32, nrhs=8, solver="mixed", precond=True),
        # S(phi) and its gradient as an autograd function, forward and backward
        dict(name="action_40", kind="action", L=40, Nt=80, nrhs=1, solver="mixed", precond=True),
        # 64 uneven chains advanced together, two right-hand sides each
        dict(name="chains_64", kind="chains", count=64, nrhs=2, guess=3, n_leap=3),
        # the benchmark's chain: multi-RHS CG with chronological starts (a short trajectory)
        dict(name="trajectory_80", kind="trajectory", L=80, Nt=160, nrhs=8, solver="mixed", precond=False, guess=4,
             n_leap=4, field="ordered"),
        # the normal operator at the benchmark's size, in the precision the inner solver runs and in FP64
        dict(name="normal_80_c64", kind="operator", op="normal", L=80, Nt=160, nrhs=8, dtype="complex64"),
        dict(name="normal_80_c128", kind="operator", op="normal", L=80, Nt=160, nrhs=8, dtype="complex128"),
        # the preconditioner at the benchmark's size
        dict(name="precond_80_c64", kind="precond", L=80, Nt=160, nrhs=8, dtype="complex64"),
        # the Fourier-diagonal velocity of one leapfrog drift
        dict(name="drift_80", kind="metric", op="velocity", L=80, Nt=160),
    ]


def _near(rng, choices, lo, hi):
    """A member of `choices` near a point spread evenly over the logarithm of [lo, hi]."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((c for c in choices if lo <= c <= hi), key=lambda c: abs(math.log(c / x)))


def draw(rng):
    kind = rng.choice(["operator", "operator", "solve", "solve", "trajectory", "precond", "metric", "action", "green",
                       "chains"])
    if kind == "chains":
        return dict(kind=kind, count=rng.randint(8, 64), nrhs=rng.choice([1, 2]), guess=rng.choice([0, 3]), n_leap=2)
    # the volume of one vector set stays within the listed extremes of its kind
    top = {"operator": 80, "precond": 80, "metric": 80, "solve": 40, "action": 40, "trajectory": 32, "green": 24}[kind]
    L = _near(rng, EXTENTS, 4, top)
    Nt = _near(rng, SLICES, 4, 2 * top)
    case = dict(kind=kind, L=L, Nt=Nt)
    if kind == "metric":
        return dict(case, op=rng.choice(["velocity", "velocity", "momentum", "kinetic"]))
    case["nrhs"] = rng.choice([1, 1, 2, 3, 4, 8])
    if kind == "operator":
        return dict(case, op=rng.choice(["normal", "normal", "D", "D_dagger"]),
                    dtype=rng.choice(["complex64", "complex128"]))
    if kind == "precond":
        return dict(case, dtype=rng.choice(["complex64", "complex64", "complex128"]))
    case["solver"] = rng.choice(["mixed", "mixed", "fp64"])
    case["precond"] = rng.random() < 0.6
    if kind == "trajectory":
        case.update(guess=rng.choice([0, 0, 3]), n_leap=rng.randint(2, 6), field="ordered")
    return case


# ---- inputs --------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(g, shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _noise(g, nrhs, L, Nt):
    """Standard complex Gaussian fermion vectors."""
    return torch.view_as_complex(_normal(g, (nrhs, Nt, L, L, 2, 2, 2))) * math.sqrt(0.5)


def _spectrum(L, Nt, r):
    """Fourier variances of the free boson, 1 / (dtau (r + kt (2 - 2 cos w) + 4 - 2 cos kx - 2 cos ky))."""
    dt, c = MODEL["dtau"], MODEL["c"]
    lap = lambda n: 2 - 2 * torch.cos(2 * math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n)
    den = r + 2.0 / (c * c * dt * dt) * lap(Nt)[:, None, None] + lap(L)[None, :, None] + lap(L)[None, None, :]
    return (1.0 / (dt * den)).expand(3, Nt, L, L).contiguous()


def _field(g, L, Nt, nrhs, r, kind="ordered"):
    z = _normal(g, (3, Nt, L, L))
    if kind == "normal":
        return z
    dims = (1, 2, 3)
    f = torch.fft.ifftn(torch.fft.fftn(z, dim=dims) * _spectrum(L, Nt, r).sqrt(), dim=dims).real.contiguous()
    f[2] += 1.2 * nrhs ** 0.4   # the mean-field amplitude: 1.2, 1.6 and 2.8 for 1, 2 and 8 right-hand sides
    return f


def _context(case, **kw):
    args = dict(MODEL, solver=case.get("solver", "mixed"), nrhs_max=case.get("nrhs", 1), cg_tol=TOL,
                initial_guess=case.get("guess", 0), **kw)
    return hmc.Context(case["L"], case["Nt"], **args)


def _chain_sizes(count, seed):
    """(L, Nt, r) of the batch: L in {12, 16, 20, 24} x Nt in {24, 32, 48}, r uniform in [0.2, 1]."""
    g = torch.Generator()
    g.manual_seed(int(seed))
    r = torch.rand(count, generator=g, dtype=torch.float64) * 0.8 + 0.2
    return [((12, 16, 20, 24)[i % 4], (24, 32, 48)[(i // 4) % 3], float(r[i])) for i in range(count)]


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "chains":
        sizes = _chain_sizes(case["count"], seed)
        L, Nt, r = sizes[0]
        ctx = hmc.Context(L, Nt, **dict(MODEL, r=r), solver="mixed", nrhs_max=case["nrhs"], cg_tol=TOL, chains=sizes,
                          initial_guess=case["guess"], batch_chains=1)
        start = torch.cat([_field(g, a, b, case["nrhs"], c).reshape(-1) for a, b, c in sizes])
        flat = start.clone()
        parts = flat.split([3 * a * a * b for a, b, _ in sizes])
        return dict(case=case, ctx=ctx, start=start, flat=flat, seed=int(seed),
                    phis=[p.view(3, b, a, a) for p, (a, b, _) in zip(parts, sizes)],
                    sigmas=[_spectrum(a, b, c) for a, b, c in sizes])
    L, Nt, nrhs = case["L"], case["Nt"], case.get("nrhs", 1)
    st = dict(case=case, ctx=_context(case))
    if kind == "metric":
        st["sigma"] = 0.15 * _spectrum(L, Nt, MODEL["r"])   # a tuned metric's ratio to the free spectrum
        pi = torch.fft.fftn(_normal(g, (3, Nt, L, L)), dim=(1, 2, 3)) / st["sigma"].sqrt()
        st["input"] = torch.fft.ifftn(pi, dim=(1, 2, 3)).real.contiguous()
        return st
    if kind == "precond":
        st["x"] = _noise(g, nrhs, L, Nt).to(getattr(torch, case["dtype"]))
        return st
    phi = _field(g, L, Nt, nrhs, MODEL["r"], case.get("field", "ordered"))
    if kind == "operator":
        st["x"] = _noise(g, nrhs, L, Nt).to(getattr(torch, case["dtype"]))
        st["phi"] = phi if case["dtype"] == "complex128" else phi.float()
    elif kind == "green":
        st["phi"] = phi
        signs = torch.randint(0, 2, (nrhs, Nt, L, L, 2, 2), generator=g, device="cuda")
        st["probes"] = (2.0 * signs.double() - 1.0).to(torch.complex128)
    elif kind in ("solve", "action"):
        st["phi"] = phi.requires_grad_(kind == "action")
        st["b"] = _noise(g, nrhs, L, Nt)
    else:
        st["start"], st["phi"] = phi, phi.clone()
        st["sigma"] = torch.ones_like(phi) if case["field"] == "normal" else 0.15 * _spectrum(L, Nt, MODEL["r"])
        st["chi"], st["z"] = _noise(g, nrhs, L, Nt), _normal(g, (3, Nt, L, L))
    return st


# ---- one pass ------------------------------------------------------------------------------------------

METRIC_OPS = {"velocity": hmc.METRIC_VELOCITY, "momentum": hmc.METRIC_MOMENTUM, "kinetic": hmc.METRIC_KINETIC}


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "operator":
        if case["op"] == "normal":
            return ctx.apply_MdagM(state["phi"], state["x"])
        return ctx.apply_M(state["phi"], state["x"], dagger=case["op"] == "D_dagger")
    if kind == "precond":
        return ctx.apply_precond(state["x"])
    if kind == "metric":
        out = ctx.metric(METRIC_OPS[case["op"]], state["sigma"], state["input"])
        return torch.tensor(out, dtype=torch.float64) if case["op"] == "kinetic" else out
    if kind == "solve":
        return ctx.cg_solve(state["phi"], state["b"], precond=case["precond"])[0]
    if kind == "green":
        return ctx.green_estimate(state["phi"], state["probes"], precond=case["precond"])[0]
    if kind == "action":
        state["phi"].grad = None
        s = pseudofermion_action(state["phi"], state["b"], ctx, precond=case["precond"])
        s.backward()
        return {"action": s.detach(), "gradient": state["phi"].grad}
    if kind == "chains":
        state["flat"].copy_(state["start"])
        o = ctx.trajectory(state["phis"], state["sigmas"], 0.02, case["n_leap"], nrhs=case["nrhs"], precond=False,
                           seed=state["seed"], counter=1)
        return {"phi": state["flat"], "energies": torch.tensor(o["energies"], dtype=torch.float64)}
    state["phi"].copy_(state["start"])
    o = ctx.trajectory([state["phi"]], [state["sigma"]], 0.05, case["n_leap"], nrhs=case["nrhs"],
                       precond=case["precond"], chi=[state["chi"]], z=[state["z"]], u=[0.0])
    return {"phi": state["phi"], "energies": torch.tensor(o["energies"], dtype=torch.float64)}


# ---- least work ----------------------------------------------------------------------------------------

def work(case):
    """Bytes: each input read once, each output written once. Flops: one D is 124 per site and right-hand
    side; a solve is counted with NOMINAL_ITERATIONS applications of D D^dagger."""
    if case["kind"] == "chains":
        V = sum(L * L * Nt for L, Nt, _ in _chain_sizes(case["count"], 0))
    else:
        V = case["L"] ** 2 * case["Nt"]
    k = case.get("nrhs", 1)
    vec, phi = 64.0 * V * k, 24.0 * V   # one complex128 vector per right-hand side, one boson field
    solve = NOMINAL_ITERATIONS * 248.0 * V * k
    kind = case["kind"]
    if kind in ("operator", "precond"):
        half = 0.5 if case["dtype"] == "complex64" else 1.0
        flops = {"normal": 248.0, "D": 124.0, "D_dagger": 124.0}.get(case.get("op"), 80.0 * math.log2(V)) * V * k
        return {"bytes": half * (2 * vec + (phi if kind == "operator" else 0)), "flops": flops}
    if kind == "metric":
        return {"bytes": 2 * phi + (0 if case["op"] == "kinetic" else phi), "flops": 15.0 * V * math.log2(V)}
    if kind == "solve":
        return {"bytes": 2 * vec + phi, "flops": solve}
    if kind == "green":
        return {"bytes": vec + 64.0 * V + phi, "flops": solve}
    if kind == "action":
        return {"bytes": vec + 2 * phi, "flops": 2 * solve}
    explicit_noise = vec + phi if kind == "trajectory" else 0.0
    return {"bytes": 3 * phi + explicit_noise, "flops": (case["n_leap"] + 1) * solve}


# ---- the same in 64 bits -------------------------------------------------------------------------------
# Vectors [k][tau][y][x][alpha][spin], fields [a][tau][y][x]: rolls along dimensions 1 to 3.

def _eta(L):
    i = torch.arange(L, device="cuda")
    return 1.0 - 2.0 * ((i[:, None] + i[None, :]) % 2).double()


def _D(phi, v, dagger=False):
    dt, Nt, L = MODEL["dtau"], phi.shape[1], phi.shape[2]
    wrap = torch.ones(Nt, device="cuda", dtype=torch.float64)
    wrap[0 if dagger else -1] = -1.0
    out = torch.roll(v, 1 if dagger else -1, dims=1) * wrap[:, None, None, None, None]
    for a in range(2):
        w = v[..., a, :]
        out[..., a, :] += (-1.0 - dt * MODEL["mu"][a]) * w
        out[..., a, :] -= dt * MODEL["t_h"][a] * (torch.roll(w, 1, dims=3) + torch.roll(w, -1, dims=3))
        out[..., a, :] -= dt * MODEL["t_v"][a] * (torch.roll(w, 1, dims=2) + torch.roll(w, -1, dims=2))
    f = dt * MODEL["g"] * _eta(L) * phi
    up, dn = v[..., 0].flip(-1), v[..., 1].flip(-1)   # the other band's spin components
    out[..., 0] += f[2][..., None] * up + torch.complex(f[0], -f[1])[..., None] * dn
    out[..., 1] += torch.complex(f[0], f[1])[..., None] * up - f[2][..., None] * dn
    return out


def _dot(a, b):
    d = (a.conj() * b).real.flatten(1).sum(1)
    return d.view(-1, 1, 1, 1, 1, 1)


def _cg(phi, b, tol, most=4000):
    x, r = torch.zeros_like(b), b.clone()
    p, rr, stop = r.clone(), _dot(r, r), tol * tol * _dot(b, b)
    for i in range(most):
        t = _D(phi, p, dagger=True)
        alpha = rr / _dot(t, t).clamp_min(1e-300)
        x += alpha * p
        r -= alpha * _D(phi, t)
        new = _dot(r, r)
        if i % 8 == 7 and bool((new <= stop).all()):
            break
        p = r + new / rr.clamp_min(1e-300) * p
        rr = new
    return x


def _solve(phi, b):
    x = _cg(phi, b, 1e-13)
    for _ in range(2):   # refinement on the true residual
        x = x + _cg(phi, b - _D(phi, _D(phi, x, dagger=True)), 1e-3)
    return x


def _fourier(x):
    return torch.fft.fftn(x, dim=(1, 2, 3), norm="ortho")


def _back(xh):
    return torch.fft.ifftn(xh, dim=(1, 2, 3), norm="ortho").real


def _twisted(v, inverse):
    Nt = v.shape[1]
    t = torch.polar(torch.ones(Nt, device="cuda", dtype=torch.float64),
                    math.pi * torch.arange(Nt, device="cuda", dtype=torch.float64) / Nt).view(1, -1, 1, 1, 1, 1)
    if inverse:
        return torch.fft.ifftn(v, dim=(1, 2, 3), norm="ortho") * t
    return torch.fft.fftn(v * t.conj(), dim=(1, 2, 3), norm="ortho")


def _precond(x):
    k, Nt, L = x.shape[:3]
    c = torch.cos(2 * math.pi * torch.arange(L, device="cuda", dtype=torch.float64) / L)
    w = (2 * torch.arange(Nt, device="cuda", dtype=torch.float64) + 1) * math.pi / Nt
    P = torch.empty(Nt, L, L, 2, device="cuda", dtype=torch.float64)
    for a in range(2):
        e = MODEL["mu"][a] + 2 * MODEL["t_h"][a] * c[None, :] + 2 * MODEL["t_v"][a] * c[:, None]
        P[..., a] = 1 / ((torch.cos(w)[:, None, None] - 1 - MODEL["dtau"] * e) ** 2 + torch.sin(w)[:, None, None] ** 2)
    return _twisted(_twisted(x, False) * P[..., None], True)


def _pf_force(phi, b):
    """-dS_PF/dphi and S_PF."""
    X = _solve(phi, b)
    Y = _D(phi, X, dagger=True).flip(-2)   # the other band
    x0, x1, y0, y1 = X[..., 0].conj(), X[..., 1].conj(), Y[..., 0], Y[..., 1]
    parts = ((x0 * y1 + x1 * y0).real, (x0 * y1 - x1 * y0).imag, (x0 * y0 - x1 * y1).real)
    F = torch.stack([p.sum(dim=(0, 4)) for p in parts])
    return 2 * MODEL["dtau"] * MODEL["g"] * _eta(phi.shape[2]) * F, float(_dot(b, X).sum())


def _boson(phi):
    """-dS_B/dphi and S_B."""
    dt, kt = MODEL["dtau"], 1.0 / (MODEL["c"] * MODEL["dtau"]) ** 2
    r, u, q = MODEL["r"], MODEL["u"], (phi * phi).sum(0)
    up = [torch.roll(phi, -1, dims=d) - phi for d in (1, 2, 3)]
    lap = [torch.roll(v, 1, dims=d) - v for v, d in zip(up, (1, 2, 3))]
    S = dt * float(kt * (up[0] ** 2).sum() + 0.5 * ((up[1] ** 2).sum() + (up[2] ** 2).sum() + (r * q).sum())
                   + 0.25 * u * (q * q).sum())
    return -dt * (2 * kt * lap[0] + lap[1] + lap[2] + (r + u * q) * phi), S


def exact(case, seed):
    kind = case["kind"]
    if kind == "chains":
        return None   # 64 chains' solves take minutes here
    V = case["L"] ** 2 * case["Nt"]
    if kind == "trajectory" and V * case["nrhs"] * case["n_leap"] > 300000:
        return None   # the benchmark's size: its solves alone take over 20 seconds
    st = prepare(case, seed)
    if kind == "operator":
        phi, x = st["phi"].double(), st["x"].to(torch.complex128)
        if case["op"] == "normal":
            x = _D(phi, x, dagger=True)
        return _D(phi, x, dagger=case["op"] == "D_dagger")
    if kind == "precond":
        return _precond(st["x"].to(torch.complex128))
    if kind == "metric":
        xh, s = _fourier(st["input"]), st["sigma"]
        if case["op"] == "kinetic":
            return 0.5 * (s * xh.abs() ** 2).sum()
        return _back(xh * (s if case["op"] == "velocity" else 1 / s.sqrt()))
    if kind == "solve":
        return _solve(st["phi"], st["b"])
    if kind == "green":
        v = st["probes"]
        u = _solve(st["phi"], _twisted(v, True))
        return (v * _twisted(_D(st["phi"], u, dagger=True), False)).mean(0)
    if kind == "action":
        F, s = _pf_force(st["phi"].detach(), st["b"])
        return {"action": torch.tensor(s, dtype=torch.float64), "gradient": -F}
    phi, sigma, eps, n = st["start"], st["sigma"], 0.05, case["n_leap"]
    pf = _D(phi, st["chi"])
    pi = _back(_fourier(st["z"]) / sigma.sqrt())
    kinetic = lambda p: float(0.5 * (sigma * _fourier(p).abs() ** 2).sum())
    before = [kinetic(pi), _boson(phi)[1], float(_dot(st["chi"], st["chi"]).sum())]
    for i in range(n + 1):
        if i:
            phi = phi + eps * _back(sigma * _fourier(pi))
        (F, s_pf), (Fb, s_b) = _pf_force(phi, pf), _boson(phi)
        pi = pi + (eps if 0 < i < n else 0.5 * eps) * (F + Fb)
    return {"phi": phi, "energies": torch.tensor([before + [kinetic(pi), s_b, s_pf]], dtype=torch.float64)}
