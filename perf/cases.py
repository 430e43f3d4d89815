"""The work users have this library do, as timed cases: new media set up and solved, many
sources on one factorisation, the preconditioner inside a caller's own iteration, and the
misfit gradient, over the sizes, precisions and options in use.

Sizes and options come from the library's own workloads (n = 64, 127, 255, 511, 1023; 16
points per wavelength for the weakly admissible format, 8 for the strongly admissible one;
PML of 8 to 16 cells; eps_H = 1e-6, or 1e-9 on the smallest grid).  Media and sources are
synthetic.  Every case ends in a converged wavefield or gradient, so its outputs do not depend
on how the approximate inverse inside is rounded.  Mixed-precision results are kept as
complex64 (float32 for the gradient), the precision such a program asked for.
"""
import math

import torch

import paper_1007_4290_gb300 as hs

DEVICE = "cuda"
TWO_PI = 2.0 * math.pi


def _case(name, kind, n, nrhs, prec, **kw):
    c = dict(name=name, kind=kind, n=n, nrhs=nrhs, prec=prec, strong=0, medium="random", medium_seed=1, ppw=16,
             pml=12, eps_H=1e-6, tol=1e-8, steps=0, dir=1)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one vector on the 64 x 64 constant-velocity grid in FP64, the
        # preconditioner inside the caller's own defect correction (launches and latency)
        _case("iterate_n64_fp64_1", "iterate", 64, 1, "fp64", medium="const", pml=8, eps_H=1e-9, steps=4),
        # a medium that changes from call to call (one step of an inversion): factor, one solve
        _case("setup_n127_mixed", "setup", 127, 1, "mixed", pml=8),
        _case("setup_n511_mixed", "setup", 511, 1, "mixed", medium="lens"),
        # the same in FP64 on a ragged grid
        _case("setup_n150_fp64", "setup", 150, 1, "fp64", pml=8, tol=1e-11),
        # the strongly admissible format of the paper's experiments (R = 2, 8 points a wavelength)
        _case("setup_strong_n255_mixed", "setup", 255, 1, "mixed", strong=2, medium="lens", ppw=8, pml=8),
        # the headline: 64 sources on one factorisation of the n = 1023 random medium
        _case("solve_n1023_mixed_64", "solve", 1023, 64, "mixed", pml=16, tol=1e-7),
        # one source at a time at n = 511
        _case("solve_n511_mixed_1", "solve", 511, 1, "mixed", medium="lens"),
        # a ragged grid with a ragged batch, swept from x2 = 1 downward
        _case("solve_down_n700_mixed_10", "solve", 700, 10, "mixed", pml=16, dir=-1),
        # FP64 end to end
        _case("solve_n255_fp64_4", "solve", 255, 4, "fp64", pml=8, tol=1e-11),
        # strongly admissible factors, several sources
        _case("solve_strong_n511_mixed_16", "solve", 511, 16, "mixed", strong=2, medium="lens", ppw=8, pml=8),
        # the preconditioner in the caller's own iteration on a batch of 64
        _case("iterate_n511_mixed_64", "iterate", 511, 64, "mixed", medium="lens", steps=3),
        # the misfit and its gradient for 32 sources and a line of receivers
        _case("grad_n511_mixed_32", "grad", 511, 32, "mixed", medium="lens"),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["setup", "solve", "solve", "iterate", "grad"])
    prec = "fp64" if rng.random() < 0.25 else "mixed"
    strong = 2 if prec == "mixed" and rng.random() < 0.25 else 0
    if prec == "fp64":
        top = 150 if kind == "setup" else 255
    else:
        top = 511 if kind in ("setup", "grad") or strong else 1023
    if kind == "setup" and strong:
        top = 255
    n = _log_int(rng, 48, top)
    nrhs = 1 if kind == "setup" else _log_int(rng, 1, 4 if prec == "fp64" else 64)
    medium = "lens" if strong else rng.choice(["random", "random", "lens", "const"])
    c = _case("", kind, n, nrhs, prec, strong=strong, medium=medium, medium_seed=rng.randrange(1, 1000),
              ppw=8 if strong else rng.choice([12, 16, 20]), pml=8 if strong or n < 160 else rng.choice([10, 12, 16]),
              tol=1e-11 if prec == "fp64" else rng.choice([1e-7, 1e-8]), dir=rng.choice([1, 1, 1, -1]))
    if kind == "iterate":
        c.update(steps=5 if prec == "fp64" else 3)
        if strong or prec == "fp64":
            # a rank-2 inverse contracts the defect too slowly for a fixed number of steps, and
            # FP64 accuracy takes GMRES: the caller's iteration is a solve there
            c.update(kind="solve", steps=0)
    del c["name"]
    return c


# ---- inputs ------------------------------------------------------------------------------


def _generator(seed):
    g = torch.Generator()
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _medium(case, seed):
    """(n, n) float64 velocity on the device, rows x2."""
    n = case["n"]
    g = _generator(seed)
    h = 1.0 / (n + 1)
    x = (torch.arange(n, dtype=torch.float64) + 1.0) * h
    if case["medium"] == "const":
        c = torch.full((n, n), 1.0 + 0.1 * (torch.rand((), generator=g, dtype=torch.float64).item() - 0.5),
                       dtype=torch.float64)
        return c.to(DEVICE)
    if case["medium"] == "lens":
        j = 0.1 * (torch.rand(2, generator=g, dtype=torch.float64) - 0.5)
        r2 = (x[None, :] - 0.5 - j[0]) ** 2 + (x[:, None] - 0.5 - j[1]) ** 2
        return ((4.0 / 3.0) * (1.0 - 0.5 * torch.exp(-32.0 * r2))).to(DEVICE)
    # a random smooth medium: filtered noise, correlation length 32 cells (two wavelengths)
    g0 = torch.randn(n, n, generator=g, dtype=torch.float64).to(DEVICE)
    t = torch.arange(n, dtype=torch.float64, device=DEVICE)
    k = torch.exp(-0.5 * ((t[:, None] - t[None, :]) / 32.0) ** 2)
    f = k @ g0 @ k.t()
    f = (f - f.mean()) / f.std()
    return 1.0 + 0.2 * f.clamp(-3.0, 3.0)


def _omega(case):
    return TWO_PI * (case["n"] + 1) / case["ppw"]


def _sources(case, seed):
    """(nrhs, n*n) complex128: discrete deltas (mass one, a random phase) inside the PML; for
    the gradient on the line x2 = 0.9."""
    n, k = case["n"], case["nrhs"]
    g = _generator(seed + 1000003)
    eta = (case["pml"] + 1) / (n + 1)
    p = eta + (1.0 - 2.0 * eta) * torch.rand(k, 2, generator=g, dtype=torch.float64)
    if case["kind"] == "grad":
        p[:, 1] = 0.9 if 0.9 < 1.0 - eta else 1.0 - 1.5 * eta
    ph = torch.rand(k, generator=g, dtype=torch.float64) * TWO_PI
    idx = torch.clamp(torch.floor(p * (n + 1) + 0.5).long() - 1, 0, n - 1)
    amp = torch.polar(torch.full((k,), float((n + 1) ** 2), dtype=torch.float64), ph)
    f = torch.zeros(k, n * n, dtype=torch.complex128, device=DEVICE)
    f[torch.arange(k, device=DEVICE), (idx[:, 1] * n + idx[:, 0]).to(DEVICE)] = amp.to(DEVICE)
    return f, p


def _receivers(case):
    n = case["n"]
    row = max(0, min(n - 1, int(math.floor(0.85 * (n + 1) + 0.5)) - 1))
    return row * n + torch.arange(n, dtype=torch.int32, device=DEVICE)


def _recorded(case, p, seed):
    """Stand-in for recorded data: the far field of a constant medium with a little noise."""
    n = case["n"]
    om = _omega(case)
    x = (torch.arange(n, dtype=torch.float64) + 1.0) / (n + 1)
    r = torch.sqrt((x[None, :] - p[:, :1]) ** 2 + (0.85 - p[:, 1:]) ** 2) + 1e-3
    d = 0.25 * torch.polar(torch.sqrt(2.0 / (math.pi * om * r)), om * r - 0.75 * math.pi)
    noise = torch.randn(p.shape[0], n, 2, generator=_generator(seed + 2000003), dtype=torch.float64)
    return (d + 0.01 * torch.view_as_complex(noise)).to(DEVICE)


def _opts(case):
    return hs.default_opts(precision=hs.FP64 if case["prec"] == "fp64" else hs.MIXED, strong_rank=case["strong"],
                           sweep_dir=case["dir"])


def _factor(case, c):
    return hs.hsweep_setup(c, _omega(case), case["pml"], case["eps_H"], _opts(case))


_kept = {}   # the factorisation in use: a program solves many batches of sources with one


def _handle(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "kind", "nrhs", "tol", "steps")))
    if key not in _kept:
        _kept.clear()
        c = _medium(case, case["medium_seed"])
        _kept[key] = (_factor(case, c), c)
    return _kept[key]


def prepare(case, seed):
    f, p = _sources(case, seed)
    if case["kind"] == "setup":
        return dict(case=case, f=f, c=_medium(case, seed))
    h, c = _handle(case)
    s = dict(case=case, f=f, h=h)
    if case["kind"] == "grad":
        s.update(rec=_receivers(case), d=_recorded(case, p, seed))
    return s


def run(state):
    case, f = state["case"], state["f"]
    mixed = case["prec"] == "mixed"
    if case["kind"] == "setup":
        h = _factor(case, state["c"])
        u, _, _ = hs.hsweep_solve(h, f, case["tol"])
        h.free()
    elif case["kind"] == "solve":
        u, _, _ = hs.hsweep_solve(state["h"], f, case["tol"])
    elif case["kind"] == "iterate":
        h = state["h"]
        u = hs.hsweep_apply(h, f)
        for _ in range(case["steps"]):
            u += hs.hsweep_apply(h, f - hs.hsweep_matvec(h, u))
    else:
        J, g = hs.hsweep_grad(state["h"], f, state["rec"], state["d"], case["tol"])
        return [J, g.float() if mixed else g]
    return [u.to(torch.complex64) if mixed else u]


# ---- what the work needs, and what it gives --------------------------------------------------


def work(case):
    """One pass: inputs read once (sources, data, and the factors, about 18 columns a depth), the
    outputs written once; operations of one apply per right-hand side (two for a gradient), and for
    a setup those of the rank-18 products of one inversion per layer."""
    n, k = case["n"], case["nrhs"]
    N = n * n
    L = max(1, math.ceil(math.log2(n / 8.0)))
    es = 8 if case["prec"] == "mixed" else 16
    per_row = (24 + 6 * (L - 1)) if case["strong"] else 8 + 18 * L
    factors = N * per_row * es
    vec = N * k * 16
    out = N * k * es
    apply_flops = 8.0 * k * 2 * N * ((24 + 12 * (L - 1)) if case["strong"] else 8 + 36 * L)
    if case["kind"] == "grad":
        return {"bytes": vec + n * k * 16 + factors + N * es // 2, "flops": 2 * apply_flops}
    if case["kind"] == "setup":
        return {"bytes": N * 8 + vec + factors + out, "flops": apply_flops + 24.0 * N * (18 * L) ** 2}
    return {"bytes": vec + factors + out, "flops": apply_flops}


def _operator(case, c):
    """The 5-point operator with its PML (sigma = 2 pi / eta (t / eta)^2): diagonal, and the edge
    coefficients towards x1 and x2, complex128."""
    n = case["n"]
    om = _omega(case)
    h = 1.0 / (n + 1)
    eta = case["pml"] * h

    def stretch(t):
        lo = ((t - eta) / eta) ** 2 * (t < eta)
        hi = ((t - 1.0 + eta) / eta) ** 2 * (t > 1.0 - eta)
        return 1.0 / torch.complex(torch.ones_like(t), (TWO_PI / eta) * (lo + hi) / om)

    node = stretch((torch.arange(n, dtype=torch.float64, device=DEVICE) + 1.0) * h)
    half = stretch((torch.arange(n + 1, dtype=torch.float64, device=DEVICE) + 0.5) * h)
    east = half[None, :] / node[:, None] / h ** 2          # (n, n + 1)
    north = half[:, None] / node[None, :] / h ** 2         # (n + 1, n)
    s12 = node[None, :] * node[:, None]
    diag = om * om / (c * c) / s12 - (east[:, :-1] + east[:, 1:] + north[:-1] + north[1:])
    return diag, east, north, s12


def _direct(op, n):
    """u = A^{-1} f by block elimination from both ends to the middle layer, all in complex128."""
    diag, east, north, _ = op
    mid = n // 2
    eye = torch.arange(n, device=DEVICE)

    def layer(m):
        S = torch.zeros(n, n, dtype=torch.complex128, device=DEVICE)
        S[eye, eye] = diag[m]
        S[eye[:-1], eye[1:]] = east[m, 1:n]
        S[eye[1:], eye[:-1]] = east[m, 1:n]
        return S

    T = [None] * n
    lo, hi = -1, n
    while lo + 1 < mid or hi - 1 > mid:
        todo = []
        if lo + 1 < mid:
            lo += 1
            S = layer(lo)
            if lo > 0:
                S -= north[lo][:, None] * T[lo - 1] * north[lo][None, :]
            todo.append((lo, S))
        if hi - 1 > mid:
            hi -= 1
            S = layer(hi)
            if hi < n - 1:
                S -= north[hi + 1][:, None] * T[hi + 1] * north[hi + 1][None, :]
            todo.append((hi, S))
        inv = torch.linalg.inv(torch.stack([S for _, S in todo]))
        for k, (m, _) in enumerate(todo):
            T[m] = inv[k]
    S = layer(mid)
    if mid > 0:
        S -= north[mid][:, None] * T[mid - 1] * north[mid][None, :]
    if mid < n - 1:
        S -= north[mid + 1][:, None] * T[mid + 1] * north[mid + 1][None, :]
    T[mid] = torch.linalg.inv(S)

    def solve(f):
        v = f.reshape(-1, n, n).permute(1, 2, 0).contiguous()      # (layer, row, source)
        for m in range(1, mid + 1):
            v[m] -= north[m][:, None] * (T[m - 1] @ v[m - 1])
        for m in range(n - 2, mid - 1, -1):
            v[m] -= north[m + 1][:, None] * (T[m + 1] @ v[m + 1])
        v[mid] = T[mid] @ v[mid]
        for m in range(mid - 1, -1, -1):
            v[m] = T[m] @ (v[m] - north[m + 1][:, None] * v[m + 1])
        for m in range(mid + 1, n):
            v[m] = T[m] @ (v[m] - north[m][:, None] * v[m - 1])
        return v.permute(2, 0, 1).reshape(-1, n * n)

    return solve


def exact(case, seed):
    """The same outputs from the direct solution of the discrete problem in complex128."""
    if case["n"] > 800:
        return None     # the dense elimination takes too long
    f, p = _sources(case, seed)
    c = _medium(case, seed if case["kind"] == "setup" else case["medium_seed"])
    op = _operator(case, c)
    solve = _direct(op, case["n"])
    u = solve(f)
    if case["kind"] != "grad":
        return [u]
    rec = _receivers(case).long()
    res = u[:, rec] - _recorded(case, p, seed)
    J = 0.5 * (res.real ** 2 + res.imag ** 2).sum()
    b = torch.zeros_like(u)
    b[:, rec] = -res.conj()
    v = solve(b)
    g = -2.0 * _omega(case) ** 2 / c.reshape(-1) ** 3 * ((u * v).sum(0) / op[3].reshape(-1)).real
    return [J.item(), g]
