"""What a user of this framework has it do, as cases that can be timed and compared.

A case is one call (or the short sequence of calls that a program makes for one result)
through paper_2010_13289_gb300.tenom / .autograd: the operator, SSP-RK3 steps with the time
step chosen on the device, the host-buffer call, the batched 1D launch and the frozen-branch
adjoint, in 1D, 2D and 3D, with both stencils, both limiters of the workloads, periodic and
transmissive boundaries, from a 256-cell shock tube (launch latency) to a 256^3 box.

States are drawn on the device from the seed, shaped like the workloads of
paper_2010_13289_gb300/problems.py.  exact() restates the method in plain 64-bit torch.
"""
import math
from fractions import Fraction

import numpy as np
import torch

from paper_2010_13289_gb300 import autograd as AG
from paper_2010_13289_gb300 import tenom as T

GAMMA = 1.4
LIMITERS = {"mp": T.LIM_MP, "tvd5": T.LIM_TVD5}
LE_BLANC_GAMMA = 5.0 / 3.0


# ------------------------------------------------------------------------------- the cases
def _grid_case(name, call, nx, ny, nz, K, lim, bc, flow, steps=1, positivity=False):
    return {"name": name, "call": call, "nx": nx, "ny": ny, "nz": nz, "K": K, "lim": lim, "bc": bc, "flow": flow,
            "steps": steps, "positivity": positivity}


def listed():
    return [
        # the smallest calls: a single shock tube, a few steps; launches and latency
        _grid_case("riemann_1d_256", "advance", 256, 1, 1, 6, "mp", "t", "riemann", steps=8),
        # the near-vacuum tube with the positivity limiter
        _grid_case("le_blanc_1d_900", "advance", 900, 1, 1, 8, "mp", "t", "le_blanc", steps=4, positivity=True),
        # one operator evaluation on an odd, ragged 3D block with mixed boundaries, as a
        # time integrator of the caller's own makes it
        _grid_case("rhs_3d_ragged", "rhs", 97, 61, 45, 6, "tvd5", "ptp", "waves"),
        # the two 2D benchmark workloads: one step of each
        _grid_case("broadband_2d_2048_teno6_mp", "advance", 2048, 2048, 1, 6, "mp", "pp", "broadband"),
        _grid_case("broadband_2d_2048_teno8_tvd5", "rk3", 2048, 2048, 1, 8, "tvd5", "pp", "broadband"),
        # an odd-sized 2D grid with outflow boundaries
        _grid_case("waves_2d_777x531", "advance", 777, 531, 1, 8, "mp", "tt", "waves", steps=2),
        # under-resolved turbulence (late Taylor-Green): many nonsmooth stencils
        _grid_case("turbulence_3d_64", "advance", 64, 64, 64, 8, "mp", "ppp", "turbulence"),
        # the 3D benchmark workload, the largest
        _grid_case("solenoidal_3d_256", "advance", 256, 256, 256, 8, "mp", "ppp", "solenoidal"),
        # host buffers in, host buffers out
        _grid_case("host_2d_1024", "host", 1024, 1024, 1, 6, "mp", "pp", "broadband"),
        # 512 shock tubes of uneven size, one step of all of them
        {"name": "batch_512", "call": "batch", "problems": 512, "nmin": 128, "nmax": 8192, "K": 6, "lim": "mp",
         "flow": "riemann", "positivity": False, "steps": 1},
        # the gradient of a rollout: forward, then the checkpointed reverse
        {"name": "rollout_2d_512", "call": "rollout", "nx": 512, "ny": 512, "nz": 1, "K": 6, "lim": "mp", "bc": "pp",
         "flow": "broadband", "steps": 8, "every": 4, "tape": "linear"},
        # one reverse step that records its own tape (memory-poor callers), 8-point scheme
        {"name": "reverse_2d_256", "call": "reverse", "nx": 256, "ny": 256, "nz": 1, "K": 8, "lim": "tvd5", "bc": "pt",
         "flow": "waves", "steps": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    K, lim = rng.choice((6, 8)), rng.choice(("mp", "tvd5"))
    kind = rng.choice(("1d", "2d", "3d", "batch", "reverse", "rollout"))
    if kind == "1d":
        c = _grid_case("", "advance", _log(rng, 100, 20000), 1, 1, K, lim, rng.choice("pt"),
                       rng.choice(("riemann", "waves", "le_blanc")), steps=rng.randint(2, 8))
        c["positivity"] = c["flow"] == "le_blanc"
        if c["flow"] != "waves":
            c["bc"] = "t"
    elif kind == "2d":
        c = _grid_case("", rng.choice(("advance", "rk3", "rhs", "host")), _log(rng, 40, 2048), _log(rng, 40, 2048), 1,
                       K, lim, rng.choice(("pp", "pt", "tp", "tt")), rng.choice(("broadband", "waves")))
        if c["flow"] == "broadband":
            c["bc"] = "pp"
    elif kind == "3d":
        c = _grid_case("", rng.choice(("advance", "rk3", "rhs")), _log(rng, 20, 160), _log(rng, 20, 160),
                       _log(rng, 20, 160), K, lim, "ppp", rng.choice(("solenoidal", "turbulence", "waves")))
        if c["flow"] == "waves":
            c["bc"] = "".join(rng.choice("pt") for _ in range(3))
    elif kind == "batch":
        nmin = _log(rng, 32, 512)
        c = {"call": "batch", "problems": _log(rng, 16, 512), "nmin": nmin, "nmax": nmin * rng.randint(2, 16), "K": K,
             "lim": lim, "flow": rng.choice(("riemann", "le_blanc")), "steps": rng.randint(1, 3)}
        c["positivity"] = c["flow"] == "le_blanc"
    else:
        c = {"call": kind, "nx": _log(rng, 40, 512), "ny": _log(rng, 40, 512), "nz": 1, "K": K, "lim": lim,
             "bc": rng.choice(("pp", "pt", "tp", "tt")), "flow": rng.choice(("broadband", "waves")), "steps": 1}
        if c["flow"] == "broadband":
            c["bc"] = "pp"
        if kind == "rollout":
            c.update(steps=rng.randint(2, 8), every=rng.randint(2, 4), tape=rng.choice(("linear", "flags")))
    c.pop("name", None)
    return c


def _shape(case):
    """Cells per axis, x first, without the axes that the case does not have."""
    return tuple(n for n, used in zip((case["nx"], case["ny"], case["nz"]), case["bc"]) if used)


def _gamma(case):
    return LE_BLANC_GAMMA if case["flow"] == "le_blanc" else GAMMA


def _lengths(case):
    return {"solenoidal": 2.0 * math.pi, "turbulence": 2.0 * math.pi, "le_blanc": 9.0}.get(case["flow"], 1.0)


# ------------------------------------------------------------------------------ the states
def _centres(n, length=1.0):
    return (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * (length / n)


def _wavenumbers(shape):
    """Integer wavevector components (slowest axis first, halved along x as rfftn keeps them)."""
    ks = [torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda") for n in shape[:-1]]
    ks.append(torch.arange(shape[-1] // 2 + 1, dtype=torch.float64, device="cuda"))
    return torch.meshgrid(*ks, indexing="ij")


def _random_phases(gen, shape):
    return torch.fft.rfftn(torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen))


def _unit_rms(f):
    return f / f.square().mean().sqrt()


def _broadband(gen, shape):
    """Base (1, 0, 0, 1/gamma) with rms-1e-2 modes 1 <= |k| <= 32 and four discs of higher
    density and pressure (problems.broadband_2d)."""
    ks = _wavenumbers(shape)
    kk = sum(k * k for k in ks)
    mask = (kk >= 1.0) & (kk <= min(32, min(shape) // 4) ** 2)
    prim = []
    for base in (1.0, 0.0, 0.0, 1.0 / GAMMA):
        spec = _random_phases(gen, shape)
        f = 1e-2 * _unit_rms(torch.fft.irfftn(torch.where(mask, spec / spec.abs().clamp_min(1e-300), 0.0 * spec), s=shape))
        prim.append(base * (1.0 + f) if base else f)
    y, x = torch.meshgrid(*[_centres(n) for n in shape], indexing="ij")
    for cx, cy, r, q in torch.rand((4, 4), dtype=torch.float64, device="cuda", generator=gen).tolist():
        dx, dy = (x - cx).abs(), (y - cy).abs()
        inside = torch.minimum(dx, 1.0 - dx) ** 2 + torch.minimum(dy, 1.0 - dy) ** 2 < (0.05 + 0.1 * r) ** 2
        ratio = torch.where(inside, 2.0 + 8.0 * q, 1.0)
        prim[0], prim[3] = prim[0] * ratio, prim[3] * ratio
    return torch.stack(prim)


def _vortical(gen, shape, spectrum):
    """Solenoidal random-phase velocity of unit rms speed with the energy spectrum E(k)."""
    ks = _wavenumbers(shape)  # z, y, x
    kk = sum(k * k for k in ks)
    k = kk.sqrt().clamp_min(1e-30)
    amp = torch.where(kk > 0, (spectrum(k) / kk.clamp_min(1e-30)).sqrt(), 0.0 * kk)
    comps = [amp * _random_phases(gen, shape) for _ in range(3)]  # x, y, z
    kd = sum(kv * c for kv, c in zip(reversed(ks), comps)) / kk.clamp_min(1e-30)
    vel = [torch.fft.irfftn(c - kv * kd, s=shape) for kv, c in zip(reversed(ks), comps)]
    rms = sum(v.square().mean() for v in vel).sqrt()
    return [v / rms for v in vel]


def _solenoidal(gen, shape):
    """rho = 1, p = 1/gamma, E(k) ~ k^4 exp(-2 (k/4)^2), rms Mach 0.6 (problems.solenoidal_3d)."""
    vel = _vortical(gen, shape, lambda k: k ** 4 * torch.exp(-2.0 * (k / 4.0) ** 2))
    one = torch.ones(shape, dtype=torch.float64, device="cuda")
    return torch.stack([one] + [0.6 * v for v in vel] + [one / GAMMA])


def _turbulence(gen, shape):
    """An inertial range down to the grid scale, E(k) ~ k^-5/3, rms Mach 0.3, with 3 %
    density and pressure fluctuations of the same spectrum."""
    vel = _vortical(gen, shape, lambda k: torch.where(k < min(shape) / 3.0, k ** (-5.0 / 3.0), 0.0 * k))
    scal = _vortical(gen, shape, lambda k: torch.where(k < min(shape) / 3.0, k ** (-5.0 / 3.0), 0.0 * k))
    return torch.stack([1.0 + 0.03 * scal[0]] + [0.3 * v for v in vel] + [(1.0 + 0.03 * scal[1]) / GAMMA])


def _waves(gen, shape):
    """A few long waves in every variable and three discs (balls, intervals) with jumps
    (problems.random_state)."""
    D = len(shape)
    r = torch.rand((D + 2, 4, D + 2), dtype=torch.float64, device="cuda", generator=gen).tolist()
    xs = torch.meshgrid(*[_centres(n) for n in shape], indexing="ij")
    prim = []
    for q in range(D + 2):
        f = torch.zeros(shape, dtype=torch.float64, device="cuda")
        for m in r[q]:
            arg = sum((1 + int(3 * m[d])) * xs[d] for d in range(D))
            f += (0.05 + 0.15 * m[D]) * torch.sin(2.0 * math.pi * (arg + m[D + 1]))
        prim.append(1.0 + 0.5 * f if q in (0, D + 1) else f)
    for c in torch.rand((3, 2 * D + 3), dtype=torch.float64, device="cuda", generator=gen).tolist():
        inside = sum((xs[d] - c[d]) ** 2 for d in range(D)) < (0.1 + 0.2 * c[D]) ** 2
        prim[0] = prim[0] * torch.where(inside, 2.0 + 4.0 * c[D + 1], 1.0)
        prim[D + 1] = prim[D + 1] * torch.where(inside, 2.0 + 4.0 * c[D + 2], 1.0)
        for d in range(D):
            prim[1 + d] = prim[1 + d] + torch.where(inside, c[D + 3 + d] - 0.5, 0.0)
    return torch.stack(prim)


def _tube(rng, n, flow):
    """(rho, u, p) of a shock tube: the Sod/Lax-like draw of problems.riemann_states, or the
    Le Blanc states with the left pressure and right density scaled by up to 20 %."""
    if flow == "le_blanc":
        a, b = rng.uniform(0.8, 1.2, 2)
        left, right, xc = (1.0, 0.0, a / 15.0), (1e-3 * b, 0.0, 2e-10 / 3.0), 1.0 / 3.0
    else:
        rho, u, p = rng.uniform(0.1, 1.0, 2), rng.uniform(-1.0, 1.0, 2), rng.uniform(0.1, 1.0, 2)
        left, right, xc = (rho[0], u[0], p[0]), (rho[1], u[1], p[1]), 0.5
    m = (np.arange(n) + 0.5) / n < xc
    return np.stack([np.where(m, a, b) for a, b in zip(left, right)])


def _primitives(case, seed):
    shape = tuple(reversed(_shape(case)))
    if case["flow"] in ("riemann", "le_blanc"):
        return torch.from_numpy(_tube(np.random.default_rng(seed), shape[0], case["flow"])).cuda()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return {"broadband": _broadband, "solenoidal": _solenoidal, "turbulence": _turbulence,
            "waves": _waves}[case["flow"]](gen, shape).contiguous()


def _conserved(prim, gamma):
    D = prim.shape[0] - 2
    m = [prim[0] * prim[1 + d] for d in range(D)]
    ke = sum(m[d] * prim[1 + d] for d in range(D))
    return torch.stack([prim[0]] + m + [prim[D + 1] / (gamma - 1.0) + 0.5 * ke])


def _dt(case, U):
    """A step at CFL 0.4 of U, as a plain number (the time step of a rollout is fixed)."""
    D = U.dim() - 1
    g = _gamma(case)
    u = [U[1 + d] / U[0] for d in range(D)]
    p = (g - 1.0) * (U[D + 1] - 0.5 * sum(U[1 + d] * u[d] for d in range(D)))
    c = (g * p / U[0]).sqrt()
    return 0.4 / float(sum((u[d].abs() + c) * (n / _lengths(case)) for d, n in enumerate(_shape(case))).max())


def _batch_inputs(case, seed):
    sizes = np.random.default_rng(case["problems"])  # the case fixes the sizes, the seed the states
    n = np.rint(np.exp(sizes.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["problems"]))).astype(np.int32)
    rng = np.random.default_rng(seed)
    prim = np.concatenate([_tube(rng, int(k), case["flow"]) for k in n], axis=1)
    return n, _lengths(case) / n, prim


# --------------------------------------------------------------------- preparing and running
def _scheme(case):
    kw = {}
    if case["flow"] == "le_blanc":  # the paper's choice for this problem: minmod curvature, beta = 1
        kw = {"mp_curv": T.CURV_MM, "mp_beta": 1.0}
    if case.get("positivity"):
        kw["positivity"] = T.PP_ON
    return T.make_scheme(case["K"], limiter=LIMITERS[case["lim"]], **kw)


def prepare(case, seed):
    s = {"case": case, "call": case["call"]}
    if case["call"] == "batch":
        n, dx, prim = _batch_inputs(case, seed)
        s["solver"] = T.Batch(n, dx, _scheme(case), gamma=_gamma(case))
        s["U0"] = s["solver"].init_state(torch.from_numpy(prim).cuda())
        s["U"] = s["U0"].clone()
        s["solver"].set_tiling(128, 4)  # what the autotuner keeps for batches of this kind
        return s
    shape = _shape(case)
    s["solver"] = T.Solver(shape, tuple(_lengths(case) / n for n in shape),
                           tuple(T.BC_PERIODIC if b == "p" else T.BC_TRANSMISSIVE for b in case["bc"]),
                           _scheme(case), gamma=_gamma(case))
    s["U0"] = _conserved(_primitives(case, seed), _gamma(case))
    s["U"] = s["U0"].clone()
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    if case["call"] == "rk3":
        s["dt"] = torch.full((1,), _dt(case, s["U0"]), dtype=torch.float64, device="cuda")
    elif case["call"] == "host":
        s["host_in"] = s["U0"].cpu().pin_memory()
        s["host_out"] = torch.empty_like(s["host_in"]).pin_memory()
    elif case["call"] == "rollout":
        s["dt"] = _dt(case, s["U0"])
        s["w"] = torch.randn(s["U0"].shape, dtype=torch.float64, device="cuda", generator=gen)
    elif case["call"] == "reverse":
        s["dt"] = torch.full((1,), _dt(case, s["U0"]), dtype=torch.float64, device="cuda")
        s["w"] = torch.randn(s["U0"].shape, dtype=torch.float64, device="cuda", generator=gen)
        s["out"] = torch.empty_like(s["U0"])
    elif case["call"] == "rhs":
        s["out"] = torch.empty_like(s["U0"])
    return s


def run(s):
    case, S, call = s["case"], s["solver"], s["call"]
    if call == "rhs":
        return S.rhs(s["U0"], out=s["out"])
    if call == "host":
        t = S.advance_host(s["host_in"], s["host_out"], nsteps=case["steps"])
        return s["host_out"], t
    if call == "rollout":
        U0 = s["U0"].clone().requires_grad_(True)
        U = AG.rollout(U0, S, s["dt"], case["steps"], checkpoint_every=case["every"], tape=case["tape"])
        U.backward(s["w"])
        return U.detach(), U0.grad
    if call == "reverse":
        return S.rk3_step_adjoint(s["U0"], s["dt"], s["w"], out=s["out"])
    s["U"].copy_(s["U0"])  # every pass starts from the initial state
    if call == "batch":
        return S.step(s["U"], nsteps=case["steps"])
    if call == "rk3":
        return S.rk3_step(s["U"], s["dt"])
    S.t.zero_()
    return S.advance(s["U"], case["steps"]), S.t


def work(case):
    """Bytes: the state read once and written once a step (a reverse step: two states read, one
    written).  Flops, per face, RK stage and axis: the K-point flux combination, and per
    characteristic field and split side the projected differences, the smoothness
    indicators and the cutoff; per cell the fluxes and the stage combination.  A reverse
    step adds the transposed flux combination and Jacobian to a forward step."""
    K = case["K"]
    if case["call"] == "batch":
        nv, D = 3, 1
        r = math.log(case["nmax"] / case["nmin"])
        cells = case["problems"] * (case["nmax"] - case["nmin"]) / r
    else:
        D = len(_shape(case))
        nv, cells = D + 2, float(np.prod(_shape(case)))
    face = 2 * K * nv + nv * 2 * (2 * nv * (K - 1) + (75 if K == 6 else 190))
    stage = cells * (D * face + D * 3 * nv + 6 * nv)
    stages = 1 if case["call"] == "rhs" else 3 * case["steps"]
    flops, nbytes = stage * stages, 16.0 * nv * cells * (1 if case["call"] == "rhs" else case["steps"])
    if case["call"] in ("rollout", "reverse"):
        back = cells * D * (2 * K * nv + 2 * nv * nv)
        flops += stages * back + (stage * stages if case["call"] == "rollout" else 0)
        nbytes += 24.0 * nv * cells * case["steps"]
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------- the method in plain 64-bit torch
# Cell-average polynomials on the cells lo..hi about cell i, from exact rationals.
def _poly(lo, hi):
    """Coefficient matrix C: p(x) = sum_m x^m sum_j C[m][j] v_{lo+j}, cell i = [-1/2, 1/2]."""
    n = hi - lo + 1
    A = []
    for j in range(n):
        a, b = Fraction(2 * (lo + j) - 1, 2), Fraction(2 * (lo + j) + 1, 2)
        A.append([(b ** (m + 1) - a ** (m + 1)) / (m + 1) for m in range(n)] + [Fraction(int(k == j)) for k in range(n)])
    for c in range(n):  # Gauss-Jordan
        p = next(r for r in range(c, n) if A[r][c] != 0)
        A[c], A[p] = A[p], A[c]
        A[c] = [x / A[c][c] for x in A[c]]
        for r in range(n):
            if r != c and A[r][c] != 0:
                A[r] = [x - A[r][c] * y for x, y in zip(A[r], A[c])]
    return [row[n:] for row in A]


def _face_value(lo, hi):
    """Weights of v_lo..v_hi in p(1/2)."""
    C = _poly(lo, hi)
    return [float(sum(C[m][j] * Fraction(1, 2) ** m for m in range(len(C)))) for j in range(len(C))]


def _indicator(lo, hi):
    """beta = sum_{r >= 1} int (p^(r))^2 over cell i, as a symmetric form in the differences
    v_{j+1} - v_j, j = lo..hi-1."""
    C = _poly(lo, hi)
    n = len(C)
    B = [[Fraction(0)] * n for _ in range(n)]
    for r in range(1, n):
        f = [Fraction(math.factorial(m), math.factorial(m - r)) if m >= r else Fraction(0) for m in range(n)]
        for a in range(r, n):
            for b in range(r, n):
                e = a + b - 2 * r
                if e % 2:
                    continue
                w = f[a] * f[b] * 2 * Fraction(1, 2) ** (e + 1) / (e + 1)
                for j in range(n):
                    for k in range(n):
                        B[j][k] += w * C[a][j] * C[b][k]
    # v_j = v_lo + sum of differences before j
    S = [[Fraction(int(t < j)) for t in range(n - 1)] for j in range(n)]
    return [[float(sum(S[j][a] * B[j][k] * S[k][b] for j in range(n) for k in range(n))) for b in range(n - 1)]
            for a in range(n - 1)]


_STENCILS = [(-1, 1), (0, 2), (-2, 0), (0, 3), (-3, 0), (0, 4)]
_WEIGHTS = {6: [9 / 20, 6 / 20, 1 / 20, 4 / 20], 8: [3 / 7, 9 / 35, 2 / 35, 6 / 35, 1 / 70, 1 / 14]}
_CAND = [_face_value(*s) for s in _STENCILS]
_BETA = [_indicator(*s) for s in _STENCILS]
_BETA_K = {6: _indicator(-2, 3), 8: _indicator(-3, 4)}


def _form(B, d):
    """d^T B d as a sum of squares (LDL^T), which keeps its relative precision."""
    L, D = _ldl(B)
    out = 0.0
    for k in range(len(d)):
        t = d[k]
        for j in range(k + 1, len(d)):
            t = t + L[j][k] * d[j]
        out = out + D[k] * t * t
    return out


_LDL = {}


def _ldl(B):
    key = id(B)
    if key not in _LDL:
        A = np.array(B)
        n = len(A)
        L, D = np.eye(n), np.zeros(n)
        for k in range(n):
            D[k] = A[k, k]
            L[k:, k] = A[k:, k] / D[k]
            A = A - D[k] * np.outer(L[:, k], L[:, k])
        _LDL[key] = (L.tolist(), D.tolist())
    return _LDL[key]


def _minmod(*a):
    """The argument of least magnitude where all have one sign, else zero."""
    lo, hi = a[0], a[0]
    for x in a[1:]:
        lo, hi = torch.where(x < lo, x, lo), torch.where(x > hi, x, hi)
    return torch.where(lo > 0, lo, torch.where(hi < 0, hi, torch.zeros_like(lo)))


def _pick(a, b, less):
    return torch.where(b < a, b, a) if less else torch.where(b > a, b, a)


def _smooth(v, K, adaptive):
    """The cutoff decisions delta_k."""
    c = K // 2 - 1
    d = [v[t + 1] - v[t] for t in range(K - 1)]
    beta = [_form(_BETA[k], d[c + lo:c + hi]) for k, (lo, hi) in enumerate(_STENCILS[:K - 2])]
    tau = (_form(_BETA_K[K], d) - (beta[1] + beta[2] + 4.0 * beta[0]) / 6.0).abs()
    g = [(1.0 + tau / (b + 1e-40)) ** 6 for b in beta]
    ct = 1e-5
    if adaptive:
        eps = 0.9 * 0.23 / (1.0 - 0.9 * 0.23) * 1e-6
        eta = None
        for q in range(4):
            a, b = d[c + q - 1], d[c + q - 2]
            e = ((2.0 * a * b).abs() + eps) / (a * a + b * b + eps)
            eta = e if eta is None else torch.minimum(eta, e)
        m = 1.0 - torch.clamp(eta / 0.23, max=1.0)
        gm = (1.0 - m) ** 4 * (1.0 + 4.0 * m)
        ct = 10.0 ** -torch.clamp(torch.floor(10.5 - 3.5 * (1.0 - gm)), 7, 10)
    total = sum(g)
    return [x >= ct * total for x in g]


def _reconstruct(v, K, lim, opt):
    c = K // 2 - 1
    with torch.no_grad():
        keep = _smooth([x.detach() for x in v], K, K == 8)
    fk = [sum(w * v[c + lo + j] for j, w in enumerate(_CAND[k])) for k, (lo, hi) in enumerate(_STENCILS[:K - 2])]
    f, fm, fp = v[c], v[c - 1], v[c + 1]
    if lim == "tvd5":
        D = [v[c + j] - v[c + j - 1] for j in (-1, 0, 1, 2)]
        B = (-2.0 * D[0] + 11.0 * D[1] + 24.0 * D[2] - 3.0 * D[3]) / 30.0
        up = _pick(_pick(2.0 * D[1], 2.0 * D[2], True), B, True)
        dn = _pick(_pick(2.0 * D[1], 2.0 * D[2], False), B, False)
        zero = torch.zeros_like(f)
        flt = f + 0.5 * torch.where(D[1] > 0, _pick(zero, up, False), torch.where(D[1] < 0, _pick(zero, dn, True), zero))
        fk = [torch.where(s, x, flt) for s, x in zip(keep, fk)]
    else:
        d = [v[c + j + 1] - 2.0 * v[c + j] + v[c + j - 1] for j in (-1, 0, 1)]
        if opt["mm"]:
            hp, hm = _minmod(d[1], d[2]), _minmod(d[0], d[1])
        else:
            hp = _minmod(4.0 * d[1] - d[2], 4.0 * d[2] - d[1], d[1], d[2])
            hm = _minmod(4.0 * d[0] - d[1], 4.0 * d[1] - d[0], d[0], d[1])
        ul, md = f + 1.25 * (f - fm), 0.5 * (f + fp) - 0.5 * hp
        lc = f + 0.5 * (f - fm) + opt["mp_beta"] / 3.0 * hm
        lo = _pick(_pick(_pick(f, fp, True), md, True), _pick(_pick(f, ul, True), lc, True), False)
        hi = _pick(_pick(_pick(f, fp, False), md, False), _pick(_pick(f, ul, False), lc, False), True)
        fk = [torch.where(s, x, x + _minmod(lo - x, hi - x)) for s, x in zip(keep, fk)]
    return sum(w * x for w, x in zip(_WEIGHTS[K], fk))


def _faces(U, axis, case):
    """Face fluxes [nv][..., n_a + 1 along the axis, last] of U ([nv][axes x first])."""
    K, g = case["K"], _gamma(case)
    h, nv = K // 2, U.shape[0]
    D = nv - 2
    n = U.shape[1 + axis]
    j = torch.arange(-h, n + h, device=U.device)
    j = j % n if case["bc"][axis] == "p" else j.clamp(0, n - 1)
    X = U.movedim(1 + axis, -1)[..., j]
    u = [X[1 + d] / X[0] for d in range(D)]
    p = (g - 1.0) * (X[-1] - 0.5 * sum(X[1 + d] * u[d] for d in range(D)))
    cs, sr, H, un = (g * p / X[0]).sqrt(), X[0].sqrt(), (X[-1] + p) / X[0], u[axis]
    F = [X[1 + axis]] + [X[1 + d] * un + (p if d == axis else 0.0) for d in range(D)] + [(X[-1] + p) * un]

    def at(a, q):  # stencil point q of every face
        return a[..., q:q + n + 1]

    sl, srr = at(sr, h - 1), at(sr, h)
    w = 1.0 / (sl + srr)
    ut = [(sl * at(x, h - 1) + srr * at(x, h)) * w for x in u]
    Ht = (sl * at(H, h - 1) + srr * at(H, h)) * w
    q2 = sum(x * x for x in ut)
    c2 = (g - 1.0) * (Ht - 0.5 * q2)
    c = c2.sqrt()
    b1 = (g - 1.0) / c2
    b2 = 0.5 * q2 * b1
    speed = [(un - cs).abs(), un.abs(), (un + cs).abs()]
    alpha = []
    for lam in speed:
        a = at(lam, 0)
        for q in range(1, K):
            a = _pick(a, at(lam, q), False)
        alpha.append(a)
    one, zero = torch.ones_like(c), torch.zeros_like(c)
    tang = [d for d in range(D) if d != axis]
    fields = []  # (left vector, right vector, alpha)
    for sg, al in ((1.0, alpha[0]), (-1.0, alpha[2])):
        left = [0.5 * (b2 + sg * ut[axis] / c)] + [0.5 * (-b1 * ut[d] - (sg / c if d == axis else 0.0)) for d in range(D)] + [0.5 * b1]
        right = [one] + [ut[d] - (sg * c if d == axis else 0.0) for d in range(D)] + [Ht - sg * ut[axis] * c]
        fields.append((left, right, al))
    fields.append(([1.0 - b2] + [b1 * x for x in ut] + [-b1], [one] + ut + [0.5 * q2], alpha[1]))
    for t in tang:
        fields.append(([-ut[t]] + [one if d == t else zero for d in range(D)] + [zero],
                       [zero] + [one if d == t else zero for d in range(D)] + [ut[t]], alpha[1]))
    opt = {"mm": case["flow"] == "le_blanc", "mp_beta": 1.0 if case["flow"] == "le_blanc" else 4.0}
    out = [0.0] * nv
    for left, right, al in fields:
        W = [sum(x * at(X[i], q) for i, x in enumerate(left)) for q in range(K)]
        G = [sum(x * at(F[i], q) for i, x in enumerate(left)) for q in range(K)]
        fp = _reconstruct([0.5 * (G[q] + al * W[q]) for q in range(K)], K, case["lim"], opt)
        fm = _reconstruct([0.5 * (G[q] - al * W[q]) for q in reversed(range(K))], K, case["lim"], opt)
        out = [o + r * (fp + fm) for o, r in zip(out, right)]
    return torch.stack(out)


def _limited(F, U, axis, case, dt):
    """The positivity limiter on the faces F of one axis ([nv][..., faces]) for a stage dt."""
    g = _gamma(case)
    n, D = U.shape[1 + axis], U.shape[0] - 2
    j = torch.arange(-1, n + 1, device=U.device)
    j = j % n if case["bc"][axis] == "p" else j.clamp(0, n - 1)
    X = U.movedim(1 + axis, -1)[..., j]
    L, R = X[..., :-1], X[..., 1:]
    mu = 2.0 * D * dt * n / _lengths(case)

    def pressure(W):
        return (g - 1.0) * (W[-1] - 0.5 * sum(W[1 + d] ** 2 for d in range(D)) / W[0])

    def flux(W):
        un, p = W[1 + axis] / W[0], pressure(W)
        f = torch.stack([W[1 + axis]] + [W[1 + d] * un + (p if d == axis else 0.0) for d in range(D)] + [(W[-1] + p) * un])
        return f, un.abs() + (g * p / W[0]).sqrt()

    (fl, al), (fr, ar) = flux(L), flux(R)
    LF = 0.5 * (fl + fr - torch.maximum(al, ar) * (R - L))
    for value in (lambda W: W[0], pressure):  # density, then pressure on what the density left
        th = torch.ones_like(F[0])
        for W, s in ((L, -mu), (R, mu)):
            lf, hi = value(W + s * LF), value(W + s * F)
            eps = torch.clamp(lf, max=1e-13)
            th = torch.where(hi < eps, torch.minimum(th, (lf - eps) / (lf - hi)), th)
        F = torch.where(th < 1.0, LF + th * (F - LF), F)
    return F


def _operator(U, case, dt=None):
    """L(U) of U [nv][nz][ny][nx]; with dt the face fluxes are limited for that stage."""
    D = U.dim() - 1
    X = U.permute(0, *range(D, 0, -1))  # axes x first
    out = 0.0
    for a in range(D):
        F = _faces(X, a, case)
        if dt is not None and case.get("positivity"):
            F = _limited(F, X, a, case, dt)
        out = out - ((F[..., 1:] - F[..., :-1]) * (X.shape[1 + a] / _lengths(case))).movedim(-1, 1 + a)
    return out.permute(0, *range(D, 0, -1))


def _stages(U, dt, case):
    U1 = U + dt * _operator(U, case, dt)
    U2 = 0.75 * U + 0.25 * (U1 + dt * _operator(U1, case, dt))
    return U1, U2, U / 3.0 + 2.0 / 3.0 * (U2 + dt * _operator(U2, case, dt))


def _transposed(U, w, case):
    """L'(U)^T w with the branches as they fall at U."""
    with torch.enable_grad():
        X = U.detach().clone().requires_grad_(True)
        return torch.autograd.grad(_operator(X, case), X, w)[0]


def _reverse(U, dt, w, case):
    """(dU^{n+1}/dU^n)^T w of one SSP-RK3 step."""
    U1, U2, _ = _stages(U, dt, case)
    a2 = 2.0 / 3.0 * w
    a2 = a2 + dt * _transposed(U2, a2, case)
    a1 = 0.25 * a2
    a1 = a1 + dt * _transposed(U1, a1, case)
    return w / 3.0 + 0.75 * a2 + a1 + dt * _transposed(U, a1, case)


def exact(case, seed):
    call = case["call"]
    with torch.no_grad():
        if call == "batch":
            n, _, prim = _batch_inputs(case, seed)
            if len(n) * case["steps"] > 100:
                return None  # the tubes run one by one here: minutes
            out, at = [], 0
            for k in n:
                sub = {**case, "bc": "t", "nx": int(k), "ny": 1, "nz": 1}
                U = _conserved(torch.from_numpy(prim[:, at:at + k]).cuda(), _gamma(case))
                for _ in range(case["steps"]):
                    U = _stages(U, _dt(sub, U), sub)[2]
                out.append(U)
                at += int(k)
            return torch.cat(out, dim=1)
        U0 = _conserved(_primitives(case, seed), _gamma(case))
        if call == "rhs":
            return _operator(U0, case)
        if call in ("rollout", "reverse"):
            w = torch.randn(U0.shape, dtype=torch.float64, device="cuda",
                            generator=torch.Generator(device="cuda").manual_seed(seed + 1))
            dt = _dt(case, U0)
            if call == "reverse":
                return _reverse(U0, dt, w, case)
            Us = [U0]
            for _ in range(case["steps"]):
                Us.append(_stages(Us[-1], dt, case)[2])
            for U in reversed(Us[:-1]):
                w = _reverse(U, dt, w, case)
            return Us[-1], w
        U, t = U0, 0.0
        for _ in range(case["steps"]):
            dt = _dt(case, U)
            U, t = _stages(U, dt, case)[2], t + dt
        if call == "host":
            return U.cpu(), t
        if call == "rk3":
            return U
        return U, torch.full((1,), t, dtype=torch.float64, device="cuda")
