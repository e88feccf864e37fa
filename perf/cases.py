"""What a program has this library do, as measurable cases.

A case is one pass through the public entry points of ``paper_0904_4152_gb300.hn`` as a user's
program makes it: Poisson solves from the smallest grids to the largest in each precision, coefficient
kind and boundary, alone, in a batch and through the server; a solve on an operator that has just
changed; the vector operations of a solver of the user's own; and the shallow-water prediction step.

``listed()`` are the fixed cases, ``draw()`` gives further ones of the same ranges, ``prepare()`` what
the program holds before the call, ``run()`` one pass, ``work()`` what a pass cannot do without and
``exact()`` the result in 64-bit arithmetic, by plain PyTorch.
"""
import numpy as np
import torch

from paper_0904_4152_gb300 import hn

PREC = {"fp64": hn.HN_PREC_FP64, "fp32": hn.HN_PREC_FP32_DC, "fp16": hn.HN_PREC_FP16BAND_DC}
SOLVER = {"mg": hn.HN_SOLVER_MG, "pcg": hn.HN_SOLVER_PCG}
ALL_SIDES = hn.HN_DIRICHLET_ALL
LEFT_RIGHT = hn.HN_DIRICHLET_LEFT | hn.HN_DIRICHLET_RIGHT


def _solve(name, L, prec, coef="one", rhs="random", **more):
    case = {"name": name, "kind": "solve", "L": L, "prec": prec, "solver": "mg", "coef": coef, "sigma": 1.0,
            "rhs": rhs, "sides": ALL_SIDES, "tol": 1e-8, "memory": "device", "guess": False}
    case.update(more)
    return case


def listed():
    return [
        # the smallest grid in use: one FP64 solve of a smooth load, where latency is all there is
        _solve("solve_fp64_L6", 6, "fp64", rhs="smooth"),
        # a time step of a host program on a small grid: numpy in and out, the last step's solution as guess
        _solve("warm_fp32_L8_host", 8, "fp32", rhs="smooth", memory="host", guess=True),
        # the benchmark grid of a million unknowns in plain FP64 and in mixed precision
        _solve("solve_fp64_L10", 10, "fp64"),
        _solve("solve_fp32_L10", 10, "fp32"),
        # walls left and right, free top and bottom, an inhomogeneous material: CG with one FP32 cycle
        _solve("pcg_fp32_L11_sides", 11, "fp32", coef="lognormal", sides=LEFT_RIGHT, solver="pcg"),
        # the largest configured grid with a lognormal coefficient, in both storage precisions
        _solve("solve_fp32_L12", 12, "fp32", coef="lognormal"),
        _solve("solve_fp16_L12", 12, "fp16", coef="lognormal"),
        # many uneven grids in one call, the result of a parameter study's parallel stage
        {"name": "batch_fp32_256", "kind": "batch", "count": 256, "lo": 5, "hi": 9, "prec": "fp32", "levels": 0},
        # requests of all sizes that arrive together at the server
        {"name": "serve_fp32_24", "kind": "serve", "count": 24, "lo": 6, "hi": 11, "prec": "fp32", "levels": 0},
        # the coefficient changes with every step (a nonlinear material): assembly, hierarchy, solve
        _solve("rebuild_fp32_L9", 9, "fp32", coef="lognormal", kind="rebuild", memory="host"),
        # the vector work of one step of a user's own Krylov method on the library's operator
        {"name": "krylov_fp64_L11", "kind": "krylov", "L": 11, "coef": "lognormal", "sigma": 1.0, "alpha": 0.37},
        # the shallow-water prediction step on the benchmark's largest grid
        {"name": "swe_fp32_4096", "kind": "swe", "dtype": "fp32", "nx": 4096, "ny": 4096, "source": True},
    ]


def draw(rng):
    fixed = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        case = _draw(rng)
        if case not in fixed:
            return case


def _draw(rng):
    kind = rng.choice(["solve"] * 6 + ["batch", "serve", "rebuild", "krylov", "swe", "swe"])
    prec = rng.choice(["fp32", "fp32", "fp16", "fp64"])
    if kind in ("solve", "rebuild"):
        # FP64 up to the level whose solve costs what the largest listed solve does
        L = rng.randint(5, 10 if kind == "rebuild" else (11 if prec == "fp64" else 12))
        coef = rng.choice(["one", "lognormal"]) if kind == "solve" else "lognormal"
        case = _solve("", L, prec, coef=coef, rhs=rng.choice(["random", "smooth"]), kind=kind,
                      sigma=round(rng.uniform(0.5, 1.2), 3), sides=rng.choice([ALL_SIDES, LEFT_RIGHT, rng.randint(1, 15)]),
                      solver=rng.choice(["mg", "mg", "pcg"]), tol=rng.choice([1e-6, 1e-8, 1e-8]),
                      memory="host" if kind == "rebuild" else rng.choice(["device", "device", "host"]))
        del case["name"]
        if kind == "solve" and coef == "one" and case["sides"] == ALL_SIDES and case["rhs"] == "smooth":
            case["guess"] = rng.choice([False, True])
        return case
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(8, 200), "lo": rng.randint(5, 6), "hi": rng.randint(7, 9),
                "prec": rng.choice(["fp32", "fp32", "fp16"]), "levels": rng.randrange(1000)}
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(8, 20), "lo": rng.randint(6, 7), "hi": rng.randint(8, 11),
                "prec": rng.choice(["fp32", "fp16"]), "levels": rng.randrange(1000)}
    if kind == "krylov":
        return {"kind": kind, "L": rng.randint(6, 11), "coef": rng.choice(["one", "lognormal"]),
                "sigma": round(rng.uniform(0.5, 1.2), 3), "alpha": round(rng.uniform(-2, 2), 3)}
    nx, ny = (int(round(2 ** rng.uniform(6, 11.9))) for _ in range(2))
    return {"kind": kind, "dtype": rng.choice(["fp32", "fp32", "fp64"]), "nx": nx, "ny": ny, "source": rng.choice([True, True, False])}


# ------------------------------------------------------------------------------------------ inputs
def _n(L):
    return (1 << L) + 1


def _levels(case):
    """The levels of a batch or of a burst of requests (part of the case, not of its inputs)."""
    r = np.random.RandomState(case["levels"])
    return [int(v) for v in r.randint(case["lo"], case["hi"] + 1, case["count"])]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _lognormal(g, L, sigma):
    """Cell coefficients exp(sigma * field): a smooth unit-variance Gaussian field, correlation length 0.1."""
    u = _uniform(g, 3, 512)
    r = torch.sqrt(-2.0 * torch.log1p(-u[0])) / 0.1
    wx, wy, ph = r * torch.cos(2 * np.pi * u[1]), r * torch.sin(2 * np.pi * u[1]), 2 * np.pi * u[2]
    c = (torch.arange(1 << L, device="cuda", dtype=torch.float64) + 0.5) / (1 << L)
    ax, ay = torch.outer(wx, c) + ph[:, None], torch.outer(wy, c)
    f = torch.cos(ay).T @ torch.cos(ax) - torch.sin(ay).T @ torch.sin(ax)
    return torch.exp(sigma * (2.0 / 512) ** 0.5 * f)


def _unknowns(L, sides):
    m = torch.ones(_n(L), _n(L), device="cuda", dtype=torch.float64)
    if sides & 1:
        m[0] = 0
    if sides & 2:
        m[:, -1] = 0
    if sides & 4:
        m[-1] = 0
    if sides & 8:
        m[:, 0] = 0
    return m


def _problem(seed, L, coef, sigma, rhs, sides):
    """(cell coefficients or None, right-hand side, a guess near the solution or None) on the GPU."""
    g = _gen(seed)
    a = _lognormal(g, L, sigma) if coef == "lognormal" else None
    n, guess = _n(L), None
    if rhs == "random":
        b = 2 * _uniform(g, n, n) - 1
    else:                    # a few sine modes; with a = 1 between zero walls, nearly those of the solution
        t = torch.arange(n, device="cuda", dtype=torch.float64) / (n - 1)
        k = torch.arange(1, 5, device="cuda", dtype=torch.float64)
        s = torch.sin(np.pi * k[:, None] * t)
        w = (2 * _uniform(g, 4, 4) - 1) / (k[:, None] ** 2 + k ** 2)
        guess = s.T @ w @ s * _unknowns(L, sides)
        near = w * (1 + 0.05 * (2 * _uniform(g, 4, 4) - 1))      # the load has moved on since the guess
        b = s.T @ (near * np.pi ** 2 * (k[:, None] ** 2 + k ** 2)) @ s / (n - 1) ** 2
    return a, b * _unknowns(L, sides), guess


def _host(t):
    return None if t is None else np.ascontiguousarray(t.reshape(-1).cpu().numpy())


def _request(case, seed, j, L):
    return _problem(seed * 1000 + j, L, "lognormal", 1.0, "random", ALL_SIDES)


class State:
    """What the program keeps between its calls; its handles go with it."""

    def __init__(self, case):
        self.case, self.mgs, self.server = case, [], None

    def hierarchy(self, L, a, sides, **opts):
        A = hn.hn_band_create_bc(L, a, sides)
        try:
            self.mgs.append(hn.hn_mg_setup(A, **opts))
        finally:
            hn.hn_band_destroy(A)

    def __del__(self):
        for mg in self.mgs:
            hn.hn_mg_destroy(mg)
        if self.server is not None:
            hn.hn_server_destroy(self.server)
        if getattr(self, "band", None) is not None:
            hn.hn_band_destroy(self.band)


def _opts(case):
    return {"prec": PREC[case["prec"]], "solver": SOLVER[case.get("solver", "mg")], "tol": case.get("tol", 1e-8)}


SWE_OFFSETS = lambda nx: [[-2, -1, 1, 2], [-2 * nx, -nx, nx, 2 * nx], [-1, 0, 1, 2], [-nx - 1, -nx + 1, nx - 1, nx + 1]]  # noqa: E731


def prepare(case, seed):
    s = State(case)
    kind = case["kind"]
    if kind in ("solve", "rebuild"):
        L = case["L"]
        a, b, guess = _problem(seed, L, case["coef"], case["sigma"], case["rhs"], case["sides"])
        s.a = _host(a)
        # a device guess is copied into x on the stream that the solve runs on
        s.stream = torch.cuda.Stream() if case["guess"] and case["memory"] == "device" else None
        if kind == "solve":
            s.hierarchy(L, s.a, case["sides"], stream=s.stream, **_opts(case))
        put = _host if case["memory"] == "host" else lambda t: t.reshape(-1).contiguous()
        s.b = put(b)
        s.guess = put(guess) if case["guess"] else None
        s.x = np.zeros_like(s.b) if case["memory"] == "host" else torch.zeros_like(s.b)
    elif kind == "batch":
        s.levels, s.bs, s.xs = _levels(case), [], []
        sizes = [_n(L) ** 2 for L in s.levels]
        starts = np.cumsum([0] + [v + v % 2 for v in sizes])           # 16-byte aligned slices of one buffer
        s.x = torch.zeros(int(starts[-1]), device="cuda", dtype=torch.float64)
        for j, L in enumerate(s.levels):
            a, b, _ = _request(case, seed, j, L)
            s.hierarchy(L, _host(a), ALL_SIDES, **_opts(case))
            s.bs.append(b.reshape(-1).contiguous())
            s.xs.append(s.x[int(starts[j]):int(starts[j]) + sizes[j]])
    elif kind == "serve":
        s.levels = _levels(case)
        s.requests = [tuple(_host(t) for t in _request(case, seed, j, L)[:2]) for j, L in enumerate(s.levels)]
        s.server = hn.hn_server_create(40 << 30, 32)
    elif kind == "krylov":
        a, b, _ = _problem(seed, case["L"], case["coef"], case["sigma"], "random", ALL_SIDES)
        s.band = hn.hn_band_create(case["L"], _host(a))
        g = _gen(seed + 1)
        s.b = b.reshape(-1).contiguous()
        inside = _unknowns(case["L"], ALL_SIDES).reshape(-1)
        s.x, s.p, s.y0 = ((2 * _uniform(g, s.b.numel()) - 1) * inside for _ in range(3))
        s.y, s.r = torch.empty_like(s.b), torch.empty_like(s.b)
        s.scalars = torch.zeros(3, 2, device="cuda", dtype=torch.float64)    # 16 bytes each
    else:
        dt = torch.float32 if case["dtype"] == "fp32" else torch.float64
        n, g = case["nx"] * case["ny"], _gen(seed)
        s.offsets = SWE_OFFSETS(case["nx"])
        make = lambda: torch.rand(n, generator=g, device="cuda", dtype=dt)  # noqa: E731
        s.bands = [[make() - 0.5 for _ in range(4)] for _ in range(4)]
        s.u, s.v, s.w = make(), make(), make()
        s.source = make() if case["source"] else None
        s.out = torch.empty_like(s.u)
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "solve":
        if s.stream is not None:
            with torch.cuda.stream(s.stream):
                s.x.copy_(s.guess)
        elif s.guess is not None:
            s.x[:] = s.guess
        x, stats, status = hn.hn_mg_solve(s.mgs[0], case["L"], s.b, s.x, s.guess is not None)
        return {"x": x, "status": status}
    if kind == "rebuild":
        A = hn.hn_band_create_bc(case["L"], s.a, case["sides"])
        mg = hn.hn_mg_setup(A, **_opts(case))
        x, stats, status = hn.hn_mg_solve(mg, case["L"], s.b, s.x)
        hn.hn_mg_destroy(mg)
        hn.hn_band_destroy(A)
        return {"x": x, "status": status}
    if kind == "batch":
        xs, stats, status = hn.hn_mg_solve_batch(s.mgs, s.levels, s.bs, s.xs)
        return {"x": s.x, "status": status}
    if kind == "serve":
        opts = hn.hn_mg_opts_default(**_opts(case))
        tickets = [hn.hn_mg_submit(s.server, L, b, a, opts) for L, (a, b) in zip(s.levels, s.requests)]
        done = [hn.hn_mg_poll(s.server, t, L) for L, t in zip(s.levels, tickets)]
        return {"x": [x for _, x, _ in done], "status": max(status for status, _, _ in done)}
    if kind == "krylov":
        s.y.copy_(s.y0)
        norm, dot, nrm = s.scalars[0, :1], s.scalars[1, :1], s.scalars[2, :1]
        hn.hn_band_defect_norm_static(s.band, s.x, s.b, s.r, norm)
        hn.hn_dot(s.r, s.p, dot)
        hn.hn_axpy(case["alpha"], s.p, s.y)
        hn.hn_nrm2(s.y, nrm)
        return {"r": s.r, "y": s.y, "norm": norm, "dot": dot, "nrm": nrm}
    hn.hn_swe_predict(s.offsets, s.bands, s.u, s.v, s.w, s.source, s.out)
    return {"u": s.out}


def work(case):
    """Bytes: the FP64 operator, right-hand side and solution once (a rebuild: the coefficients in place
    of the operator).  Operations: nine V(2,2) cycles, five nine-point products each on a hierarchy of 4/3."""
    kind = case["kind"]
    solve = lambda L, read: (8 * (read + 2) * _n(L) ** 2, 9 * 5 * 18 * 4 / 3 * _n(L) ** 2)  # noqa: E731
    if kind in ("solve", "rebuild"):
        b, f = solve(case["L"], 9 if kind == "solve" else 1)
    elif kind in ("batch", "serve"):
        b, f = (sum(v) for v in zip(*(solve(L, 9 if kind == "batch" else 1) for L in _levels(case))))
    elif kind == "krylov":
        n = _n(case["L"]) ** 2
        b, f = n * (96 + 16 + 24 + 8), n * (20 + 2 + 2 + 2)
    else:
        n, e = case["nx"] * case["ny"], 4 if case["dtype"] == "fp32" else 8
        b, f = n * e * (20 + case["source"]), 33 * n
    return {"bytes": b, "flops": f}


# ------------------------------------------------------- the results in 64-bit arithmetic (PyTorch)
def _shift(x, dy, dx):
    """x moved so that node (y, x) holds its neighbour (y + dy, x + dx); zero off the grid."""
    n = x.shape[-1]
    return torch.nn.functional.pad(x, (1, 1, 1, 1))[..., 1 + dy:1 + dy + n, 1 + dx:1 + dx + n]


def _bands(a, mask):
    """The nine bands of the bilinear operator for cell coefficients a (..., 2^L, 2^L)."""
    p = torch.nn.functional.pad(a, (1, 1, 1, 1))
    sw, se, nw, ne = p[..., :-1, :-1], p[..., :-1, 1:], p[..., 1:, :-1], p[..., 1:, 1:]
    rows = [-sw / 3, -(sw + se) / 6, -se / 3, -(sw + nw) / 6, (sw + se + nw + ne) * (2 / 3), -(se + ne) / 6,
            -nw / 3, -(nw + ne) / 6, -ne / 3]
    out = []
    for k, v in enumerate(rows):
        if k != 4:
            v = v * mask * _shift(mask, k // 3 - 1, k % 3 - 1)
        else:
            v = torch.where(mask > 0, v, torch.ones_like(v))
        out.append(v)
    return out


def _apply(bands, x):
    y = bands[4] * x
    for k in (0, 1, 2, 3, 5, 6, 7, 8):
        y += bands[k] * _shift(x, k // 3 - 1, k % 3 - 1)
    return y


def _prolong(e, n):
    f = e.new_zeros(*e.shape[:-2], n, n)
    f[..., ::2, ::2] = e
    f[..., 1::2, ::2] = 0.5 * (e[..., 1:, :] + e[..., :-1, :])
    f[..., :, 1::2] = 0.5 * (f[..., :, 0:-1:2] + f[..., :, 2::2])
    return f


def _restrict(r):
    t = 0.5 * (_shift(r, 0, -1) + _shift(r, 0, 1)) + r
    t = 0.5 * (_shift(t, -1, 0) + _shift(t, 1, 0)) + t
    return t[..., ::2, ::2]


def _cycle(levels, k, b):
    bands, mask = levels[k]
    if k == len(levels) - 1:
        return torch.linalg.solve(bands, b.flatten(-2).unsqueeze(-1)).squeeze(-1).reshape(b.shape) * mask
    w = 0.7 / bands[4]
    x = w * b
    x += w * (b - _apply(bands, x))
    x += _prolong(_cycle(levels, k + 1, _restrict(b - _apply(bands, x)) * levels[k + 1][1]), b.shape[-1]) * mask
    for _ in range(2):
        x += w * (b - _apply(bands, x))
    return x


def _reference(L, a, b, sides):
    """The solution of A x = b to the accuracy of 64-bit arithmetic: conjugate gradients preconditioned
    by a V cycle, for a stack of problems of one level (a: (k, 2^L, 2^L), b: (k, n, n))."""
    levels = []
    for l in range(L, 1, -1):
        mask = _unknowns(l, sides)
        bands = _bands(a, mask)
        if l == 2:
            eye = torch.eye(25, device="cuda", dtype=torch.float64).reshape(25, 1, 5, 5)
            bands = _apply([v.unsqueeze(0) for v in bands], eye.expand(25, a.shape[0], 5, 5))
            bands = bands.reshape(25, -1, 25).permute(1, 2, 0)
        levels.append((bands, mask))
        a = 0.25 * (a[..., ::2, ::2] + a[..., ::2, 1::2] + a[..., 1::2, ::2] + a[..., 1::2, 1::2])
    dot = lambda u, v: (u * v).sum((-2, -1), keepdim=True)  # noqa: E731
    x, r = torch.zeros_like(b), b.clone()
    p, rz = torch.zeros_like(b), None
    for _ in range(60):
        if bool((dot(r, r) <= 1e-28 * dot(b, b)).all()):
            break
        z = _cycle(levels, 0, r)
        new = dot(r, z)
        p = z + (0 if rz is None else new / rz) * p
        q = _apply(levels[0][0], p)
        alpha = new / dot(p, q)
        x += alpha * p
        r -= alpha * q
        rz = new
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "rebuild"):
        L = case["L"]
        a, b, _ = _problem(seed, L, case["coef"], case["sigma"], case["rhs"], case["sides"])
        a = torch.ones(1 << L, 1 << L, device="cuda", dtype=torch.float64) if a is None else a
        x = _reference(L, a.unsqueeze(0), b.unsqueeze(0), case["sides"]).reshape(-1)
        return {"x": x.cpu().numpy() if case["memory"] == "host" else x, "status": hn.HN_OK}
    if kind in ("batch", "serve"):
        levels, xs = _levels(case), {}
        for L in sorted(set(levels)):
            js = [j for j, l in enumerate(levels) if l == L]
            for at in range(0, len(js), 16):              # 16 problems of a level at a time
                part = js[at:at + 16]
                ab = [_request(case, seed, j, L) for j in part]
                x = _reference(L, torch.stack([v[0] for v in ab]), torch.stack([v[1] for v in ab]), ALL_SIDES)
                xs.update({j: x[i].reshape(-1) for i, j in enumerate(part)})
        if kind == "serve":
            return {"x": [xs[j].cpu().numpy() for j in range(len(levels))], "status": hn.HN_OK}
        zero = torch.zeros(1, device="cuda", dtype=torch.float64)
        return {"x": torch.cat([torch.cat((xs[j], zero)) for j in range(len(levels))]), "status": hn.HN_OK}
    s = prepare(case, seed)
    if kind == "krylov":
        L, n = case["L"], _n(case["L"])
        a, b, _ = _problem(seed, L, case["coef"], case["sigma"], "random", ALL_SIDES)
        a = torch.ones(1 << L, 1 << L, device="cuda", dtype=torch.float64) if a is None else a
        r = (b - _apply(_bands(a, _unknowns(L, ALL_SIDES)), s.x.reshape(n, n))).reshape(-1)
        y = s.y0 + case["alpha"] * s.p
        return {"r": r, "y": y, "norm": r.norm().reshape(1), "dot": (r * s.p).sum().reshape(1), "nrm": y.norm().reshape(1)}
    u = s.u.double()
    out, n = u.clone(), u.numel()
    for m, x in enumerate((s.v.double(), s.w.double(), u, u)):
        for off, band in zip(s.offsets[m], s.bands[m]):
            lo, hi = max(0, -off), min(n, n - off)
            if lo < hi:
                out[lo:hi] += band[lo:hi].double() * x[lo + off:hi + off]
    return {"u": out + s.source.double() if s.source is not None else out}
