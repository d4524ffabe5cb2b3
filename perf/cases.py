"""Performance cases: the work that a user of the solver has it do, through its
public binding (paper_1612_08395_gb300.bem), from the smallest transform to the
largest solves.

Kinds of case, each with the sizes, precisions and options it is used with:
  transform   bem_convolve of a pressure field on a handle
  noalloc     bem_convolve_noalloc with a spectrum the caller holds
  setup       bem_create of a new grid and graded exponent, its spectrum, bem_destroy
  solve       a non-adhesive solve at one depth
  sweep       a load sweep (non-adhesive) or a pull-off (adhesive) over several depths
  serve       a mix of solves handed to the request server at once

Results of an FP32 transform are handed on as float32 (its precision); every
other result is FP64 or comes from an FP64-refined solve.
"""
import math

import numpy as np
import torch

from paper_1612_08395_gb300 import bem, inputs

NU = 0.3
DEV = "cuda"


def listed():
    return [
        # the transform of a small contact problem: latency and launches count
        {"name": "transform_64_fp64", "kind": "transform", "nx": 64, "ny": 64, "k": 0.5, "precision": "fp64"},
        # the allocation-free transform on a ragged grid, inside a host program's own loop
        {"name": "noalloc_200x251_fp64", "kind": "noalloc", "nx": 200, "ny": 251, "k": -0.3},
        # the FP32 transform at the size of the large load-unload sweeps
        {"name": "transform_2048_fp32", "kind": "transform", "nx": 2048, "ny": 2048, "k": 0.3, "precision": "fp32"},
        # the FP64 transform of a large rectangular grid of odd sizes
        {"name": "transform_1501x1100_fp64", "kind": "transform", "nx": 1501, "ny": 1100, "k": -0.5,
         "precision": "fp64"},
        # every served request of a new (grid, k) sets a handle up
        {"name": "setup_600", "kind": "setup", "n": 600, "k": 0.2},
        # the plain method on the small graded Hertz contact, FP64 throughout
        {"name": "hertz_64_fp64", "kind": "solve", "n": 64, "k": 0.5, "profile": "paraboloid", "depth": 0.01,
         "precision": "fp64"},
        # a flat cylindrical punch on an odd grid, FP64 throughout
        {"name": "punch_333_fp64", "kind": "solve", "n": 333, "k": 0.5, "profile": "punch", "depth": 0.01,
         "precision": "fp64"},
        # a seeded rough surface whose contact spans the grid
        {"name": "rough_2048_refine", "kind": "solve", "n": 2048, "k": 0.3, "profile": "rough", "depth": 0.0,
         "precision": "fp32_refine"},
        # the load sweep of the graded Hertz contact at 512^2, warm-started from depth to depth
        {"name": "load_512_refine", "kind": "sweep", "n": 512, "k": -0.5, "profile": "paraboloid", "d0": 0.002,
         "d1": 0.02, "steps": 10, "dgamma": 0.0, "precision": "fp32_refine"},
        # the 2048^2 pull-off: preload and the first unloading depths
        {"name": "pulloff_2048_refine", "kind": "sweep", "n": 2048, "k": 0.3, "profile": "paraboloid", "d0": 0.02,
         "d1": 0.02 - 6 * 1.1e-4, "steps": 7, "dgamma": 1e-3, "precision": "fp32_refine"},
        # one served adhesive request on an odd grid: preload, then unload to d = 0
        {"name": "pulloff_301_refine", "kind": "sweep", "n": 301, "k": 0.0, "profile": "paraboloid", "d0": 0.01,
         "d1": 0.0, "steps": 9, "dgamma": 1e-3, "precision": "fp32_refine"},
        # a batch of mixed solves through the request server
        {"name": "serve_12", "kind": "serve", "jobs": 12, "n_min": 64, "n_max": 512, "mix": 4,
         "precision": "fp32_refine"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges.  Graded exponents as in the served requests,
    away from the ends where the criterion of small contacts has no solution."""
    kind = rng.choice(["transform", "transform", "noalloc", "setup", "solve", "solve", "sweep", "sweep", "serve"])
    k = round(rng.uniform(-0.5, 0.7), 3)
    if kind == "transform":
        n = _log(rng, 16, 2048)
        ny = max(16, int(round(n * rng.uniform(0.5, 1.0)))) if rng.random() < 0.5 else n
        return {"kind": kind, "nx": n, "ny": ny, "k": k, "precision": rng.choice(["fp64", "fp32"])}
    if kind == "noalloc":
        return {"kind": kind, "nx": _log(rng, 8, 256), "ny": _log(rng, 8, 256), "k": k}
    if kind == "setup":
        return {"kind": kind, "n": _log(rng, 32, 1024), "k": k}
    if kind == "solve":
        prec = rng.choice(["fp64", "fp32_refine"])
        prof = rng.choice(["paraboloid", "punch", "rough"])
        return {"kind": kind, "n": _log(rng, 48, 400 if prec == "fp64" else 1024), "k": k, "profile": prof,
                "depth": 0.0 if prof == "rough" else round(rng.uniform(0.004, 0.02), 5), "precision": prec}
    if kind == "sweep":
        n = _log(rng, 64, 400)
        if rng.random() < 0.5:
            return {"kind": kind, "n": n, "k": k, "profile": "paraboloid", "d0": 0.002,
                    "d1": round(rng.uniform(0.006, 0.02), 5), "steps": rng.randint(3, 8), "dgamma": 0.0,
                    "precision": rng.choice(["fp64", "fp32_refine"])}
        return {"kind": kind, "n": n, "k": k, "profile": "paraboloid", "d0": 0.01,
                "d1": round(rng.uniform(0.0, 0.006), 5), "steps": rng.randint(3, 9),
                "dgamma": float("%.3g" % math.exp(rng.uniform(math.log(1e-4), math.log(3e-3)))),
                "precision": "fp32_refine"}
    return {"kind": kind, "jobs": rng.randint(3, 10), "n_min": 64, "n_max": _log(rng, 128, 512),
            "mix": rng.randrange(1 << 20), "precision": "fp32_refine"}


# ---------------------------------------------------------------------------
# Inputs

def _sides(case):
    return (case["nx"], case["ny"]) if "nx" in case else (case["n"], case["n"])


def _pressure(nx, ny, seed):
    """A contact pressure: Hertz-like domes with a rough part on a few patches, zero elsewhere."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    x = (torch.arange(nx, device=DEV, dtype=torch.float64) + 0.5) / nx
    y = (torch.arange(ny, device=DEV, dtype=torch.float64) + 0.5) / ny
    c = torch.rand(4, 3, generator=g, device=DEV, dtype=torch.float64)
    noise = torch.rand(ny, nx, generator=g, device=DEV, dtype=torch.float64)
    p = torch.zeros(ny, nx, device=DEV, dtype=torch.float64)
    for i in range(4):
        r2 = ((x[None, :] - c[i, 0]) ** 2 + (y[:, None] - c[i, 1]) ** 2) / (0.1 + 0.25 * c[i, 2]) ** 2
        p += torch.sqrt(torch.clamp(1.0 - r2, min=0.0))
    return p * (0.75 + 0.5 * noise)


def _profile(case, seed):
    """(heights, depth of a rough surface) of the seeded indenter of a case, on the host."""
    n = case["n"]
    r = np.random.Generator(np.random.PCG64(seed))
    u = r.random(4)
    if case["profile"] == "rough":
        h, rms = inputs.rough_self_affine(n, hurst=0.8, q1_over_q0=min(256.0, n / 8.0), rms_slope=0.1, seed=seed)
        return np.ascontiguousarray(h), rms
    dx = 1.0 / n
    x = inputs.centres(n, dx)
    cx, cy = 0.04 * (u[0] - 0.5), 0.04 * (u[1] - 0.5)
    r2 = (x[None, :] - cx) ** 2 + (x[:, None] - cy) ** 2
    if case["profile"] == "punch":
        a = 0.18 + 0.04 * u[2]
        # the face carries a faint waviness, as a machined one does
        face = 1e-5 * (1.0 + np.cos(9.0 * x[None, :] + 6.0 * u[3]) * np.cos(7.0 * x[:, None]))
        return np.where(r2 <= a * a, face, inputs.EXCLUDED), 0.0
    return np.ascontiguousarray(r2 / (2.0 * (0.9 + 0.2 * u[2]))), 0.0


def _opts(profile, precision):
    """Solver options: FP64 solves to 1e-12; a rough surface's many small contacts take
    more refinement sweeps until the contact set settles."""
    if precision == "fp64":
        return {"precision": precision, "tol": 1e-12}
    return {"precision": precision, "refine_sweeps": 24 if profile == "rough" else 0}


def _depths(case, rms):
    if case["kind"] == "solve":
        return np.array([rms if case["profile"] == "rough" else case["depth"]])
    return np.linspace(case["d0"], case["d1"], case["steps"])


def _serve_jobs(case, seed):
    """The seeded requests of a serve case: sides log-uniform, k ~ U[-0.5, 0.7], half adhesive."""
    r = np.random.Generator(np.random.PCG64(case["mix"]))
    jobs = []
    for i in range(case["jobs"]):
        n = int(round(math.exp(r.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        k = float(round(r.uniform(-0.5, 0.7), 3))
        adhesive = bool(r.random() < 0.5)
        rough = bool(r.random() < 0.5) and not adhesive
        dg = float(math.exp(r.uniform(math.log(1e-4), math.log(3e-3)))) if adhesive else 0.0
        sub = {"kind": "sweep" if adhesive else "solve", "n": n, "profile": "rough" if rough else "paraboloid",
               "depth": 0.01, "d0": 0.01, "d1": 0.004, "steps": 5}
        h, rms = _profile(sub, seed + 7919 * (i + 1))
        jobs.append({"n": n, "k": k, "dgamma": dg, "h": h, "d": _depths(sub, rms), "profile": sub["profile"]})
    return jobs


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    bem.load_library()
    if case["kind"] == "serve":
        # requests arrive with host arrays; the server lives as long as the program
        s.jobs = _serve_jobs(case, seed)
        for j in s.jobs:
            j["p"] = np.empty_like(j["h"])
        s.server = bem.Server(nworkers=8, hbm_budget_bytes=32 << 30)
        return s
    if case["kind"] == "setup":
        # the set-up has no array input: the request's own graded exponent is what changes
        s.k = _setup_k(case, seed)
        return s
    nx, ny = _sides(case)
    dx = 1.0 / max(nx, ny)
    if case["kind"] in ("transform", "noalloc"):
        s.p = _pressure(nx, ny, seed)
        s.u = torch.empty_like(s.p)
    else:
        h, rms = _profile(case, seed)
        s.d = _depths(case, rms)
        s.h = torch.from_numpy(h).to(DEV)
        s.p = torch.empty_like(s.h)
    handle = bem.Handle(nx, ny, dx, dx, case["k"], NU)
    if case["kind"] == "noalloc":
        s.khat = torch.from_numpy(handle.spectrum()).to(DEV)
        s.A = handle.info().compliance
        handle.close()
    else:
        s.handle = handle
    return s


def _setup_k(case, seed):
    return case["k"] + 1e-3 * np.random.Generator(np.random.PCG64(seed)).random()


def _results(p, res):
    return {"p": p, "force": np.array([r.force for r in res]), "area": np.array([r.area for r in res]),
            "count": np.array([r.contact_count for r in res], dtype=np.int64)}


def run(state):
    c = state.case
    kind = c["kind"]
    if kind == "transform":
        u = state.handle.convolve(state.p, precision=c["precision"], out=state.u)
        return u.to(torch.float32) if c["precision"] == "fp32" else u
    if kind == "noalloc":
        rc = bem.convolve_noalloc(state.khat, c["nx"], c["ny"], state.A, state.p, state.u,
                                  stream=torch.cuda.current_stream())
        if rc != bem.BEM_OK:
            raise RuntimeError("bem_convolve_noalloc: %d" % rc)
        return state.u
    if kind == "setup":
        n = c["n"]
        with bem.Handle(n, n, 1.0 / n, 1.0 / n, state.k, NU) as h:
            return h.spectrum()
    if kind == "solve":
        res, _ = state.handle.solve(state.h, float(state.d[0]), pressure_out=state.p,
                                    **_opts(c["profile"], c["precision"]))
        return _results(state.p, [res])
    if kind == "sweep":
        res, _ = state.handle.sweep(state.h, state.d, dgamma=c["dgamma"], final_pressure=state.p,
                                    **_opts(c["profile"], c["precision"]))
        return _results(state.p, res)
    tags = []
    for j in state.jobs:
        n = j["n"]
        tags.append(state.server.submit(n, n, 1.0 / n, 1.0 / n, j["k"], NU, j["h"], j["d"], dgamma=j["dgamma"],
                                        final_pressure=j["p"], **_opts(j["profile"], c["precision"])))
    done = {d["tag"]: d for d in state.server.drain()}
    return [_results(done[t]["final_pressure"], done[t]["results"]) for t in tags]


def work(case):
    """Each input read once, each output written once; 5 L log2 L flops per transform of
    L points, for iterated solves those of one transform per depth."""
    if case["kind"] == "serve":
        b = f = 0.0
        r = np.random.Generator(np.random.PCG64(case["mix"]))
        for _ in range(case["jobs"]):
            n = int(round(math.exp(r.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
            r.random(), r.random(), r.random()
            b += 16.0 * n * n
            f += 10.0 * (4.0 * n * n) * math.log2(4.0 * n * n)
        return {"bytes": b, "flops": f}
    nx, ny = _sides(case)
    pts = 4.0 * nx * ny
    fft = 5.0 * pts * math.log2(pts)  # two real transforms of the padded field
    if case["kind"] == "setup":
        return {"bytes": 8.0 * pts / 4, "flops": fft / 2}
    if case["kind"] == "noalloc":
        return {"bytes": 16.0 * nx * ny + 8.0 * pts / 4, "flops": fft}
    if case["kind"] == "transform":
        b = 4.0 if case["precision"] == "fp32" else 8.0
        return {"bytes": 2 * b * nx * ny + b * pts / 4, "flops": fft}
    return {"bytes": 16.0 * nx * ny, "flops": fft * case.get("steps", 1)}


# ---------------------------------------------------------------------------
# The same results in 64 bits, by plain torch and numpy

def _influence(k, dx, nx, ny):
    """K(di, dj), 0 <= di < nx, 0 <= dj < ny, of square elements: the integral of
    r^-(1+k) over the element.  Near the origin by the divergence theorem (the
    integrand is homogeneous: (1-k) K is the boundary integral of r^-(1+k) (r . n),
    with r = a cosh s on an edge at distance a); elsewhere tensor Gauss-Legendre."""
    near_x, near_y = min(9, nx), min(9, ny)
    K = torch.empty(ny, nx, device=DEV, dtype=torch.float64)

    def rule(n):
        x, w = np.polynomial.legendre.leggauss(n)
        return torch.tensor(x, device=DEV), torch.tensor(w, device=DEV)

    def tensor(j0, j1, i0, i1, n):
        if j1 <= j0 or i1 <= i0:
            return
        x, w = rule(n)
        a = torch.arange(i0, i1, device=DEV, dtype=torch.float64)[None, :]
        b = torch.arange(j0, j1, device=DEV, dtype=torch.float64)[:, None]
        s = torch.zeros(j1 - j0, i1 - i0, device=DEV, dtype=torch.float64)
        for q in range(n):
            for r in range(n):
                s += 0.25 * w[q] * w[r] * ((a + 0.5 * x[q]) ** 2 + (b + 0.5 * x[r]) ** 2) ** (-0.5 * (1.0 + k))
        K[j0:j1, i0:i1] = s

    mx, my = min(40, nx), min(40, ny)
    tensor(0, my, near_x, mx, 10)
    tensor(near_y, my, 0, near_x, 10)
    tensor(0, my, mx, nx, 4)
    tensor(my, ny, 0, nx, 4)
    gx, gw = np.polynomial.legendre.leggauss(60)

    def J(T):  # integral of cosh^-k from 0 to T
        return 0.5 * T * float(np.sum(gw * np.cosh(0.5 * T * (gx + 1.0)) ** -k))

    def edge(a, b0, b1):
        m = abs(a)
        return a * m ** -k * (J(math.asinh(b1 / m)) - J(math.asinh(b0 / m)))

    for j in range(near_y):
        for i in range(near_x):
            x0, x1, y0, y1 = i - 0.5, i + 0.5, j - 0.5, j + 0.5
            K[j, i] = (edge(x1, y0, y1) - edge(x0, y0, y1) + edge(y1, x0, x1) - edge(y0, x0, x1)) / (1.0 - k)
    return K * dx ** (1.0 - k)


def _compliance(k, nu=NU):
    """alpha (1 - nu^2) for E0 = c0 = 1."""
    b = math.sqrt((1.0 + k) * (1.0 - k * nu / (1.0 - nu)))
    al = (2.0 ** k * b * math.sin(0.5 * math.pi * b) * math.gamma(0.5 * (3.0 + k + b)) *
          math.gamma(0.5 * (3.0 + k - b))) / (math.sqrt(math.pi) * (1.0 + k) * math.cos(0.5 * math.pi * k) *
                                              math.gamma(2.0 + k) * math.gamma(1.0 + 0.5 * k) *
                                              math.gamma(0.5 * (1.0 - k)))
    return al * (1.0 - nu * nu)


class _Operator:
    """u = A K*p by torch's FP64 FFT on a zero-padded torus."""

    def __init__(self, k, dx, nx, ny):
        self.nx, self.ny = nx, ny
        K = _influence(k, dx, nx + 1, ny + 1)
        iy = torch.minimum(torch.arange(2 * ny), 2 * ny - torch.arange(2 * ny)).to(DEV)
        ix = torch.minimum(torch.arange(2 * nx), 2 * nx - torch.arange(2 * nx)).to(DEV)
        self.hat = _compliance(k) * torch.fft.rfft2(K[iy][:, ix])

    def __call__(self, p):
        X = torch.fft.rfft2(p, s=(2 * self.ny, 2 * self.nx)) * self.hat
        return torch.fft.irfft2(X, s=(2 * self.ny, 2 * self.nx))[:self.ny, :self.nx]


def _held(op, c, S, p, tol=1e-14, most=4000):
    """p with A (K p) + c = 0 on S and p = 0 off it, by conjugate gradients."""
    p = torch.where(S, p, 0.0)
    best, since = math.inf, 0
    g = torch.where(S, op(p) + c, 0.0)
    t = g.clone()
    G = float((g * g).sum())
    stop = tol * tol * float(c[S].square().sum())
    for _ in range(most):
        if G <= stop:
            break
        r = torch.where(S, op(t), 0.0)
        tau = G / float((t * r).sum())
        p = p - tau * t
        g = g - tau * r
        Gn = float((g * g).sum())
        t = g + (Gn / G) * t
        G = Gn
        since = 0 if G < 0.25 * best else since + 1
        best = min(best, G)
        if since > 200:
            break
    return p


def _free(op, h, d):
    """The p >= 0 with gap g = A K p + h - d >= 0 and p g = 0: constrained conjugate
    gradients, then the contact set's own equations."""
    c = h - d
    p = torch.where(c < 0, 1e-3, 0.0)
    t = torch.zeros_like(p)
    delta, G_old = 0.0, 1.0
    for _ in range(3000):
        g = op(p) + c
        on = p > 0
        G = float(torch.where(on, g * g, 0.0).sum())
        if G == 0.0:
            break
        t = torch.where(on, g + delta * (G / G_old) * t, 0.0)
        G_old = G
        r = op(t)
        tr = float(torch.where(on, r * t, 0.0).sum())
        gt = float(torch.where(on, g * t, 0.0).sum())
        if not (tr > 0 and gt > 0):
            break
        tau = gt / tr
        q = torch.where(on, torch.clamp(p - tau * t, min=0.0), p)
        over = (q == 0) & (g < 0)
        delta = 0.0 if bool(over.any()) else 1.0
        q = torch.where(over, -tau * g, q)
        eps = float((q - p).abs().sum() / q.sum())
        p = q
        if eps < 1e-13:
            break
    for _ in range(20):  # the set's own equations, until the set is the solution's
        S = p > 0
        p = _held(op, c, S, p)
        g = op(p) + c
        wrong = (S & (p < 0)) | (~S & (g < -1e-14))
        if not bool(wrong.any()):
            break
        p = torch.where(S & (p < 0), 0.0, p)
        p = torch.where(~S & (g < -1e-14), 1e-12, p)
    return p


_C1 = {0.0: 2.97, 0.3: 5.62, 0.5: 9.15, -0.5: 0.96}  # corrected c1 at tabulated exponents


def _solve_exact(case, seed):
    n = case["n"]
    dx = 1.0 / n
    h0, rms = _profile(case, seed)
    op = _Operator(case["k"], dx, n, n)
    h = torch.from_numpy(h0).to(DEV)
    cell = dx * dx
    force, area = [], []
    dg = case.get("dgamma", 0.0)
    S = p = None
    for i, d in enumerate(_depths(case, rms)):
        if dg == 0.0 or i == 0:
            p = _free(op, h, float(d))
            S = p > 0
        else:
            crit = math.sqrt(2.0 * dg / (_compliance(case["k"]) * _C1[case["k"]] * dx ** (1.0 - case["k"])))
            while True:
                p = _held(op, h - float(d), S, p, tol=1e-13)
                off = S & (-p > crit)
                if not bool(off.any()):
                    break
                S = S & ~off
                p = torch.where(S, p, 0.0)
        force.append(cell * float(p.sum()))
        area.append(cell * int(S.sum()))
    return {"p": p, "force": np.array(force), "area": np.array(area), "count": None}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("transform", "noalloc"):
        nx, ny = _sides(case)
        return _Operator(case["k"], 1.0 / max(nx, ny), nx, ny)(_pressure(nx, ny, seed))
    if kind == "setup":
        n = case["n"]
        P = 32
        while P < 2 * n:
            P *= 2
        K = _influence(_setup_k(case, seed), 1.0 / n, P // 2 + 1, P // 2 + 1)
        i = torch.minimum(torch.arange(P), P - torch.arange(P)).to(DEV)
        return torch.fft.rfft2(K[i][:, i]).real[:P // 2 + 1].cpu().numpy()
    if kind == "serve" or case["n"] > 640:
        return None
    if case.get("dgamma", 0.0) > 0.0 and (case["n"] > 160 or case["k"] not in _C1):
        return None
    return _solve_exact(case, seed)
