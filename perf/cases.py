"""Workloads of the library, for measuring it: each case is one call sequence that a user's program
makes through the package's public entry points.

A case is a dict of plain values: "kind" (what is called), nx, ny, nz (points per axis; 0: the axis
does not exist) and the options of that call.

  apply     Grid.apply of the pressure operator with a density that stays attached
  fft       Grid.fft_r2c and Grid.fft_c2r of two unrelated fields
  pressure  Grid.set_density, then Grid.solve of the pressure system (one time step's, or one request's)
  velocity  the same with the coupled velocity system
  krho      the same with the modified-Helmholtz form of the pressure system
  step      Flow.step
  batch     Batch.run: velocity and pressure systems of uneven instances in one graph launch

Densities are the ones the paper's cases have (a top-hat in 1D, a perturbed two-layer interface, slabs
three cells sharp, a swirling jet), right-hand sides smooth random fields or the divergence of a noisy
predictor velocity.  Launch shapes are the built-in ones: nothing is autotuned.
"""

import math

import torch

import paper_2403_06654_gb300 as vd

DEV = "cuda"
TWO_PI = 2.0 * math.pi


def listed():
    return [
        # one implicit 1D solve to near rounding (top-hat density): the lowest latency there is
        {"name": "pressure_1d_256_f64", "kind": "pressure", "nx": 256, "ny": 0, "nz": 0, "ratio": 3.0,
         "solver": "cg", "precision": "fp64", "tol": 1e-12},
        # a small plane's operator apply, the inner call of a user's own iteration: launches count
        {"name": "apply_2d_96_f64", "kind": "apply", "nx": 96, "ny": 96, "nz": 0, "ratio": 3.0},
        # a small request of the serving mix
        {"name": "pressure_2d_192_dd", "kind": "pressure", "nx": 192, "ny": 192, "nz": 0, "ratio": 8.0,
         "solver": "cg", "precision": "mixed_dd", "tol": 1e-10},
        # a mid-size plane of unequal lengths, high density ratio, residual kept in double
        {"name": "pressure_2d_480x360_mixed", "kind": "pressure", "nx": 480, "ny": 360, "nz": 0, "ratio": 20.0,
         "solver": "gmres", "precision": "mixed", "tol": 1e-10},
        # the velocity system of a 2D instance of the batched mix
        {"name": "velocity_2d_320_dd", "kind": "velocity", "nx": 320, "ny": 320, "nz": 0, "ratio": 6.0,
         "solver": "gmres", "precision": "mixed_dd", "tol": 1e-10},
        # one semi-implicit step of the Rayleigh-Taylor-like layer, everything in double
        {"name": "step_rt_512x1024_f64", "kind": "step", "nx": 512, "ny": 1024, "nz": 0, "ratio": 3.0,
         "precision": "fp64", "tol": 1e-10},
        # a 3D request of the serving mix, length with a factor 5, density ratio above 10
        {"name": "pressure_3d_80_dd", "kind": "pressure", "nx": 80, "ny": 80, "nz": 80, "ratio": 16.0,
         "solver": "cg", "precision": "mixed_dd", "tol": 1e-10},
        # a 3D velocity system of the batched mix
        {"name": "velocity_3d_96_dd", "kind": "velocity", "nx": 96, "ny": 96, "nz": 96, "ratio": 5.0,
         "solver": "gmres", "precision": "mixed_dd", "tol": 1e-10},
        # plain single-precision transforms of a box of unequal lengths
        {"name": "fft_3d_320x256x160_f32", "kind": "fft", "nx": 320, "ny": 256, "nz": 160, "precision": "mixed"},
        # a 3D pressure solve in plain double
        {"name": "pressure_3d_128_f64", "kind": "pressure", "nx": 128, "ny": 128, "nz": 128, "ratio": 4.0,
         "solver": "cg", "precision": "fp64", "tol": 1e-10},
        # uneven instances, velocity and pressure systems, recorded into one graph
        {"name": "batch_6_dd", "kind": "batch", "nx": 160, "ny": 160, "nz": 64, "count": 6, "ratio": 10.0,
         "precision": "mixed_dd", "tol": 1e-10},
        # the 256^3 swirling jet's pressure solve: the headline workload
        {"name": "pressure_jet_256_dd", "kind": "pressure", "nx": 256, "ny": 256, "nz": 256, "ratio": 2.0,
         "density": "jet", "solver": "cg", "precision": "mixed_dd", "tol": 1e-10},
    ]


def _smooth(rng, lo, hi):
    """An even 2-3-5-smooth length, spread over the logarithm of [lo, hi]."""
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    sizes = sorted({2 ** a * 3 ** b * 5 ** c for a in range(1, 11) for b in range(5) for c in range(4)})
    return min((s for s in sizes if lo <= s <= hi), key=lambda s: abs(math.log(s / t)))


def draw(rng):
    kind = rng.choice(["pressure", "pressure", "pressure", "velocity", "velocity", "apply", "fft", "step", "krho",
                       "batch"])
    ratio = round(math.exp(rng.uniform(math.log(2.0), math.log(20.0))), 2)
    precision = rng.choice(["mixed_dd", "mixed_dd", "mixed", "fp64"])
    if kind == "batch":
        return {"kind": kind, "nx": _smooth(rng, 64, 240), "ny": _smooth(rng, 64, 240), "nz": _smooth(rng, 32, 64),
                "count": rng.randint(2, 6), "ratio": min(ratio, 10.0), "precision": "mixed_dd", "tol": 1e-10}
    dim = 2 if kind == "step" else rng.choice([2, 3, 3])
    if kind in ("pressure", "krho") and rng.random() < 0.15:
        dim = 1
    # double runs at a fraction of the single rate and a velocity apply is worth several pressure ones: smaller boxes
    small = kind == "velocity" or precision == "fp64"
    lo, hi = {1: (64, 1024), 2: (64, 384 if small or kind == "step" else 900), 3: (32, 96 if small else 160)}[dim]
    n = [_smooth(rng, lo, hi) for _ in range(dim)] + [0] * (3 - dim)
    case = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2]}
    if kind != "fft":
        case["ratio"] = min(ratio, {"step": 4.0, "velocity": 8.0}.get(kind, 8.0 if small else 20.0))
    if kind != "apply":
        case["precision"] = precision
    if kind == "step":
        case.update(precision=rng.choice(["fp64", "mixed_dd"]), tol=1e-10)
    elif kind not in ("apply", "fft"):
        case.update(solver="gmres" if kind == "velocity" or (dim < 3 and rng.random() < 0.3) else "cg", tol=1e-10)
    return case


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------

def _n(case):
    return tuple(v for v in (case["nx"], case["ny"], case["nz"]) if v)


def _coords(n, L):
    out = []
    for j in range(len(n)):
        sh = [1] * len(n)
        sh[len(n) - 1 - j] = n[j]
        out.append((L[j] / n[j] * torch.arange(n[j], dtype=torch.float64, device=DEV)).reshape(sh))
    return out


def _uniform(gen, lo, hi):
    return lo + (hi - lo) * torch.rand((), generator=gen, dtype=torch.float64).item()


def _slab(n, L, ratio, gen):
    """Top-hat of density `ratio` across half of a random axis, interfaces about three cells wide."""
    axis = int(torch.randint(0, len(n), (), generator=gen))
    centre, thick = _uniform(gen, 0.0, L[axis]), 3.0 * L[axis] / n[axis]
    x = _coords(n, L)[axis]
    r = torch.remainder(x - centre + L[axis] / 2, L[axis]) - L[axis] / 2
    w = L[axis] / 4
    rho = 1.0 + 0.5 * (ratio - 1.0) * (torch.tanh((r + w) / thick) - torch.tanh((r - w) / thick))
    return rho.expand(tuple(reversed(n))).contiguous()


def _smooth_field(n, L, gen, kmax=5):
    """Twelve random Fourier modes with |m| <= kmax along each axis."""
    f = torch.zeros(tuple(reversed(n)), dtype=torch.float64, device=DEV)
    X = _coords(n, L)
    for _ in range(12):
        m = torch.randint(-kmax, kmax + 1, (len(n),), generator=gen).tolist()
        amp = torch.randn((), generator=gen, dtype=torch.float64).item()
        arg = sum(TWO_PI * m[j] / L[j] * X[j] for j in range(len(n))) + _uniform(gen, 0.0, TWO_PI)
        f += amp * torch.cos(arg)
    return f


def _noise(shape, seed):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    return torch.randn(shape, generator=g, dtype=torch.float64, device=DEV)


def _system(case, seed):
    """(n, L, rho, b) of a case with one density and one right-hand side."""
    gen = torch.Generator().manual_seed(int(seed))
    n = _n(case)
    L = (TWO_PI,) * len(n)
    if len(n) == 1:      # the 1D top-hat and its 16-mode right-hand side
        x = _coords(n, L)[0]
        a, d = _uniform(gen, 0.4, 0.6) * math.pi, max(0.05, 2.5 * TWO_PI / n[0])
        rho = 1.0 + 0.5 * (case["ratio"] - 1.0) * (torch.tanh((x - a) / d) - torch.tanh((x - a - math.pi) / d))
        b = torch.zeros_like(x)
        for k in range(1, 17):
            c = torch.randn(2, generator=gen, dtype=torch.float64).tolist()
            b += (c[0] * torch.cos(k * x) + c[1] * torch.sin(k * x)) / k ** 2
        return n, L, rho, b
    if len(n) == 3 and case.get("density") == "jet":
        # swirling jet: density 1/ratio inside, right-hand side the divergence of the noisy predictor velocity
        x, y, z = _coords(n, L)
        yc, zc = y - L[1] / 2 + _uniform(gen, -0.2, 0.2), z - L[2] / 2
        prof = 0.5 * (1.0 - torch.tanh((torch.sqrt(yc ** 2 + zc ** 2) - 0.5) / 0.05))
        sh = tuple(reversed(n))
        rho = (1.0 + (1.0 / case["ratio"] - 1.0) * prof).expand(sh).contiguous()
        b = torch.zeros(sh, dtype=torch.float64, device=DEV)
        for j, base in enumerate((prof, -prof * zc, prof * yc)):
            b += _d((base + 1e-3 * _noise(sh, seed * 3 + j)).contiguous(), j, n, L)
        return n, L, rho, b
    rho = _slab(n, L, case["ratio"], gen)
    if case["kind"] == "velocity":
        b = torch.stack([_smooth_field(n, L, gen) for _ in n])
    else:
        b = _smooth_field(n, L, gen)
    return n, L, rho, b


def _flow_inputs(case, seed):
    """Two fluid layers (heavy slab, its lower interface perturbed) in a box twice as high as wide, at rest
    but for 1e-3 noise."""
    n = _n(case)
    L = (1.0, 2.0)
    x, z = _coords(n, L)
    gen = torch.Generator().manual_seed(int(seed))
    eta = 0.05 * torch.cos(TWO_PI * (x + _uniform(gen, 0.0, 1.0)))
    delta = max(0.02, 6.0 / n[1])
    rho = 1.0 + 0.5 * (case["ratio"] - 1.0) * (torch.tanh((z - 0.5) / delta + eta) - torch.tanh((z - 1.5) / delta))
    return n, L, rho.contiguous(), 1e-3 * _noise((2,) + tuple(reversed(n)), seed)


FLOW = {"Re": 1000.0, "Sc": 1.0, "Fr": 1.0, "dt": 1e-3}


def _instances(case, seed):
    """Uneven instances of the batched workload: 2D and 3D in turn, sizes around the case's."""
    out = []
    for i in range(case["count"]):
        gen = torch.Generator().manual_seed(int(seed) * 64 + i)
        if i % 2:
            n = (case["nz"], case["nz"], case["nz"]) if i % 4 == 1 else (case["nz"], case["nz"], 32)
        else:
            n = (case["nx"], case["ny"]) if i % 4 == 0 else (case["ny"], case["nx"])
        L = (TWO_PI,) * len(n)
        ratio = 2.0 + (case["ratio"] - 2.0) * i / max(1, case["count"] - 1)
        out.append({"n": n, "L": L, "rho": _slab(n, L, ratio, gen), "a": 1e-3, "inv_sc": 1.0,
                    "b_vel": torch.stack([_smooth_field(n, L, gen) for _ in n]), "b_pres": _smooth_field(n, L, gen)})
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        items = _instances(case, seed)
        for it in items:
            it["x_vel"], it["x_pres"] = torch.zeros_like(it["b_vel"]), torch.zeros_like(it["b_pres"])
        B = vd.Batch(items, vel_solver="gmres", pres_solver="cg", tol=case["tol"], max_it=500, restart=30,
                     precision=case["precision"])
        return {"kind": kind, "B": B, "x": [(it["x_vel"], it["x_pres"]) for it in items]}
    if kind == "fft":
        n = _n(case)
        G = vd.Grid(n, (TWO_PI,) * len(n))
        dt = torch.float32 if case["precision"] == "mixed" else torch.float64
        sh = tuple(reversed(n))
        f, g = _noise(sh, seed).to(dt), _noise(sh, seed + (1 << 40)).to(dt)
        return {"kind": kind, "G": G, "f": f, "gh": torch.fft.rfftn(g).contiguous(), "precision": case["precision"]}
    if kind == "step":
        n, L, rho, u = _flow_inputs(case, seed)
        G = vd.Grid(n, L)
        F = vd.Flow(G, Re=FLOW["Re"], Sc=FLOW["Sc"], Fr=FLOW["Fr"], gravity_axis=1, vel_solver="rmr",
                    pres_solver="gmres", tol=case["tol"], max_it=200, restart=30, precision=case["precision"])
        F.set_state(rho, u)
        return {"kind": kind, "F": F}
    n, L, rho, b = _system(case, seed)
    G = vd.Grid(n, L)
    if kind == "apply":
        G.set_density(rho)
        return {"kind": kind, "G": G, "b": b}
    return {"kind": kind, "G": G, "rho": rho, "b": b, "solver": case["solver"], "tol": case["tol"],
            "precision": case["precision"]}


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return state["G"].apply("pressure", state["b"])
    if kind == "fft":
        G, p = state["G"], state["precision"]
        return [G.fft_r2c(state["f"], precision=p), G.fft_c2r(state["gh"], precision=p)]
    if kind == "step":
        state["F"].step(FLOW["dt"])
        return list(state["F"].state())
    if kind == "batch":
        state["B"].run()
        return state["x"]
    G = state["G"]
    G.set_density(state["rho"], op=kind)
    kw = {"a": 1e-3, "inv_sc": 1.0} if kind == "velocity" else {}
    x, _ = G.solve(kind, state["solver"], state["b"], tol=state["tol"], max_it=500, restart=30,
                   precision=state["precision"], **kw)
    return x


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------

def _iterations(ratio, tol):
    """Krylov iterations to reduce the residual by tol at condition number `ratio` (the CG bound)."""
    s = math.sqrt(max(ratio, 1.01))
    return math.log(2.0 / tol) / math.log((s + 1.0) / (s - 1.0))


def _solve_work(kind, n, ratio, tol):
    d, N = len(n), math.prod(n)
    fft = 2.5 * N * math.log2(N)            # one real transform
    if kind == "velocity":                  # V_rho: d (d + 2) inverse and d forward transforms
        return {"bytes": 8.0 * N * (1 + 2 * d), "flops": 6.0 * d * (d + 3) * fft}
    per = 2.0 if kind == "krho" else 2.0 * d
    return {"bytes": 8.0 * N * 3, "flops": _iterations(ratio, tol) * per * fft}


def work(case):
    kind, n = case["kind"], _n(case)
    N = math.prod(n)
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for i in range(case["count"]):
            m = ((case["nx"], case["ny"]) if i % 2 == 0 else
                 (case["nz"], case["nz"], case["nz"] if i % 4 == 1 else 32))
            ratio = 2.0 + (case["ratio"] - 2.0) * i / max(1, case["count"] - 1)
            for k in ("velocity", "pressure"):
                w = _solve_work(k, m, ratio, case["tol"])
                total = {key: total[key] + w[key] for key in total}
        return total
    fft = 2.5 * N * math.log2(N)
    if kind == "fft":
        return {"bytes": 4.0 * N * (4 if case["precision"] == "mixed" else 8), "flops": 2.0 * fft}
    if kind == "apply":
        return {"bytes": 8.0 * N * 3, "flops": (2 * len(n) + 2) * fft}
    if kind == "step":       # state (rho, u, grad p, phi, history) in and out, and the two solves
        v, p = (_solve_work(k, n, case["ratio"], case["tol"]) for k in ("velocity", "pressure"))
        return {"bytes": 8.0 * N * 18, "flops": v["flops"] + p["flops"]}
    return _solve_work(kind, n, case["ratio"], case["tol"])


# ---------------------------------------------------------------------------------------
# the results in 64 bits, from the definitions, with library transforms
# ---------------------------------------------------------------------------------------

def _k(j, n, L, full=False):
    """Wavenumbers along axis j of a half spectrum, shaped to broadcast; 0 at the Nyquist index unless full."""
    m = torch.arange(n[j] // 2 + 1 if j == 0 else n[j], dtype=torch.float64, device=DEV)
    m = torch.where(2 * m > n[j], m - n[j], m)
    if not full:
        m = torch.where(m.abs() * 2 == n[j], torch.zeros_like(m), m)
    sh = [1] * len(n)
    sh[len(n) - 1 - j] = m.numel()
    return (TWO_PI / L[j] * m).reshape(sh)


def _k2(n, L, full=False):
    return sum(_k(j, n, L, full) ** 2 for j in range(len(n)))


def _F(f, n):
    return torch.fft.rfftn(f, dim=tuple(range(-len(n), 0)))


def _iF(h, n):
    return torch.fft.irfftn(h, s=tuple(reversed(n)), dim=tuple(range(-len(n), 0)))


def _d(f, j, n, L):
    return _iF(1j * _k(j, n, L) * _F(f, n), n)


def _pinv(k2, sign):
    return torch.where(k2 > 0, sign / torch.where(k2 > 0, k2, torch.ones_like(k2)), torch.zeros_like(k2))


def _pressure_apply(x, rho, n, L):
    h = _F(x, n)
    return sum(_d(_iF(1j * _k(j, n, L) * h, n) / rho, j, n, L) for j in range(len(n)))


def _cg(A, M, b, tol=1e-15, most=1500):
    """Preconditioned CG on a negative semi-definite pair, until the residual no longer falls."""
    x, r = torch.zeros_like(b), b.clone()
    z = M(r)
    p, rz = z, torch.sum(r * z)
    best, at, bn = (math.inf, x), 0, torch.linalg.vector_norm(b).item()
    for it in range(most):
        q = A(p)
        alpha = rz / torch.sum(p * q)
        x = x + alpha * p
        r = r - alpha * q
        rel = torch.linalg.vector_norm(r).item() / bn
        if rel < 0.5 * best[0]:
            at = it
        if rel < best[0]:
            best = (rel, x)
        if rel <= tol or it - at > 60:
            break
        z = M(r)
        new = torch.sum(r * z)
        p, rz = z + (new / rz) * p, new
    return best[1]


def _exact_pressure(rho, b, n, L):
    k2 = _k2(n, L)
    keep = (k2 > 0).to(torch.float64)
    inv = _pinv(k2, -1.0)
    x = torch.zeros_like(b)
    b = _iF(keep * _F(b, n), n)
    for _ in range(2):      # the second solve corrects by the true residual of the first
        r = b - _pressure_apply(x, rho, n, L)
        x = x + _cg(lambda v: _pressure_apply(v, rho, n, L), lambda v: _iF(inv * _F(v, n), n), _iF(keep * _F(r, n), n))
    return _iF(keep * _F(x, n), n)


def _exact_krho(rho, b, n, L):
    k2 = _k2(n, L, full=True)
    w = rho ** -0.5
    c = _iF(k2 * _F(w, n), n) / w
    inv = _pinv(k2, -1.0)

    def A(v):
        return _iF(-k2 * _F(v, n), n) + c * v

    b = b - w * (torch.sum(w * b) / torch.sum(w * w))
    x = torch.zeros_like(b)
    for _ in range(2):
        r = b - A(x)
        r = r - w * (torch.sum(w * r) / torch.sum(w * w))
        x = x + _cg(A, lambda v: _iF(inv * _F(v, n), n), r)
    return x - x.mean()


def _velocity_apply(u, rho, n, L, a, inv_sc=1.0):
    d = len(n)
    g = [_d(rho, j, n, L) for j in range(d)]
    k2 = _k2(n, L)
    out = []
    for i in range(d):
        t = _iF(-k2 * _F(u[i], n), n)
        for j in range(d):
            t = t + inv_sc * (u[j] * _d(g[i], j, n, L) + g[j] * _d(u[i], j, n, L))
        out.append(u[i] - a * _iF(_F(t / rho, n), n))
    return torch.stack(out)


def _exact_velocity(rho, b, n, L, a, x0=None):
    """Restarted, right-preconditioned GMRES."""
    sym = 1.0 / (1.0 + a * _k2(n, L))
    x = torch.zeros_like(b) if x0 is None else x0
    bn = torch.linalg.vector_norm(b).item()
    last = math.inf
    for _ in range(12):
        r = b - _velocity_apply(x, rho, n, L, a)
        beta = torch.linalg.vector_norm(r).item()
        if beta <= 2e-15 * bn or beta > 0.5 * last:
            break
        last = beta
        V, H = [r / beta], torch.zeros(31, 30, dtype=torch.float64)
        for j in range(30):
            w = _velocity_apply(_iF(sym * _F(V[j], n), n), rho, n, L, a)
            for _ in range(2):
                for i in range(j + 1):
                    h = torch.sum(w * V[i])
                    H[i, j] += h.item()
                    w = w - h * V[i]
            H[j + 1, j] = torch.linalg.vector_norm(w).item()
            V.append(w / H[j + 1, j])
            e = torch.zeros(j + 2, 1, dtype=torch.float64)
            e[0] = beta
            y = torch.linalg.lstsq(H[:j + 2, :j + 1], e).solution
            if torch.linalg.vector_norm(H[:j + 2, :j + 1] @ y - e).item() <= 1e-9 * beta:
                break
        x = x + _iF(sym * _F(sum(y[i, 0].item() * V[i] for i in range(y.shape[0])), n), n)
    return x


def _exact_step(case, seed):
    """The first step (explicit terms by Euler) of the scheme that Flow documents."""
    n, L, rho0, u = _flow_inputs(case, seed)
    dt, Re, Sc, Fr = FLOW["dt"], FLOW["Re"], FLOW["Sc"], FLOW["Fr"]
    d, a = len(n), FLOW["dt"] / (2.0 * FLOW["Re"])
    k2 = _k2(n, L)
    c = dt / (2.0 * Re * Sc)
    adv = sum(u[j] * _d(rho0, j, n, L) for j in range(d))
    rho1 = _iF(((1.0 - c * k2) * _F(rho0, n) - dt * _F(adv, n)) / (1.0 + c * k2), n)
    rho = 0.5 * (rho0 + rho1)
    advu = torch.stack([sum(u[j] * _d(u[i], j, n, L) for j in range(d)) for i in range(d)])
    rhs = u - dt * advu + u - _velocity_apply(u, rho, n, L, a, 1.0 / Sc)
    rhs[1] += -dt / Fr * (1.0 - rho.mean() / rho)
    us = _exact_velocity(rho, rhs, n, L, a, u)
    phi = _exact_pressure(rho, sum(_d(us[j], j, n, L) for j in range(d)) / dt, n, L)
    gphi = torch.stack([_d(phi, j, n, L) for j in range(d)])
    w = gphi / rho
    q = rho * (w - _velocity_apply(w, rho, n, L, a, 1.0 / Sc))
    ph = _pinv(k2, -1.0) * _F(sum(_d(q[j], j, n, L) for j in range(d)), n)
    gp = gphi - torch.stack([_iF(1j * _k(j, n, L) * ph, n) for j in range(d)])
    return [rho1, us - dt * w, gp, phi]


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [(_exact_velocity(it["rho"], it["b_vel"], it["n"], it["L"], it["a"]),
                 _exact_pressure(it["rho"], it["b_pres"], it["n"], it["L"])) for it in _instances(case, seed)]
    if kind == "fft":
        s = prepare(case, seed)
        n = _n(case)
        gh = s["gh"].to(torch.complex128)
        return [_F(s["f"].to(torch.float64), n), _iF(gh, n)]
    if kind == "step":
        return _exact_step(case, seed)
    n, L, rho, b = _system(case, seed)
    if kind == "apply":
        return _pressure_apply(b, rho, n, L)
    if kind == "velocity":
        return _exact_velocity(rho, b, n, L, 1e-3)
    return _exact_krho(rho, b, n, L) if kind == "krho" else _exact_pressure(rho, b, n, L)
