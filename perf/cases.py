"""Performance cases of the TENO-D gas-kinetic solver, through its public Python
entry points: single 1-D tubes, 2-D planes, batches of tubes, and the adjoint.

Every case starts each pass from the same seeded state (a user's restart: set
the state, advance, read it back) and returns whole states.  A state is
float64 at the entry points.  The float64 path's states are returned as they
are; the mixed path computes its reconstructions and fluxes in float32, so its
states are returned in that type, the one its digits are good for.

`exact` is the scheme in plain torch float64, written from the paper's
formulas (moments of the Maxwellian and linear solves for the slopes).
"""
import math

import numpy as np
import torch

from paper_2309_10534_gb300 import gks

GAMMA = 1.4
EPS, Q, CT1, CT2 = 1e-40, 7, 1e-7, 1e-5  # TENO-D (the library's defaults)
D_HI, D_LO, EPS_AO = 0.85, 0.85, 1e-8    # WENO5-AO
C1, C2 = 0.01, 1.0                       # Euler collision time


def listed():
    """Sizes are those of the repository's workloads, tests and benchmark."""
    def tube(name, nx, precision, steps, **kw):
        return dict({"name": name, "kind": "tube", "nx": nx, "precision": precision, "steps": steps, "tau": "euler",
                     "recon": "teno_d", "bc": "zerograd", "call": "advance"}, **kw)

    def plane(name, nx, ny, precision, steps, **kw):
        return dict({"name": name, "kind": "plane", "nx": nx, "ny": ny, "precision": precision, "steps": steps,
                     "tau": "euler", "recon": "teno_d", "bc": "zerograd", "cfl": 0.5, "Pr": 1.0, "call": "step"}, **kw)

    return [
        # one time step for a caller that owns all device memory: the smallest call
        {"name": "noalloc_400_fp64", "kind": "noalloc", "nx": 400, "precision": "fp64"},
        # Sod's tube at the paper's 400 cells: a whole small run is hundreds of such steps
        tube("tube_400_fp64", 400, "fp64", 16),
        # shock / density-wave tubes at 1000 cells in mixed precision
        tube("tube_1000_fp32", 1000, "fp32", 24),
        # a long tube: 1-D throughput
        tube("tube_4m_fp32", 1 << 22, "fp32", 4, call="step"),
        # a coarse plane, as in parameter studies and tests
        plane("plane_64_fp32", 64, 64, "fp32", 4, call="advance"),
        # Riemann problem at the paper's 400 x 400 and CFL 0.8 in the default precision
        plane("plane_400_fp64", 400, 400, "fp64", 2, cfl=0.8),
        # the benchmark's plane, mixed precision
        plane("plane_1024_fp32", 1024, 1024, "fp32", 2),
        # the comparison reconstruction on a ragged plane
        plane("plane_333x517_ao_fp32", 333, 517, "fp32", 2, recon="weno_ao"),
        # viscous shock tube at full size: walls, Navier-Stokes collision time, Prandtl number
        plane("viscous_2048x1024_fp32", 2048, 1024, "fp32", 2, tau="ns", bc="walls", cfl=0.2, Pr=0.73),
        # many independent tubes in one launch
        {"name": "batch_1024_fp32", "kind": "batch", "count": 1024, "nmin": 200, "nmax": 4000, "precision": "fp32",
         "steps": 24},
        # gradient of a smooth flow: checkpointed forward and backward pass, kept adjoint object
        {"name": "adjoint_512_fp32", "kind": "adjoint", "nx": 512, "ny": 512, "precision": "fp32", "steps": 12,
         "every": 6, "call": "object"},
        # the differentiable map inside a small optimisation
        {"name": "flow_96_fp64", "kind": "adjoint", "nx": 96, "ny": 96, "precision": "fp64", "steps": 4, "every": 2,
         "call": "flow"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["noalloc", "tube", "tube", "plane", "plane", "plane", "batch", "adjoint"])
    precision = rng.choice(["fp64", "fp32"])
    if kind == "noalloc":
        return {"kind": kind, "nx": _log(rng, 100, 16384), "precision": precision}
    if kind == "tube":
        nx = _log(rng, 100, 1 << 22 if precision == "fp32" else 1 << 18)
        return {"kind": kind, "nx": nx, "precision": precision, "steps": rng.randint(1, 8),
                "tau": rng.choice(["euler", "euler", "zero"]),
                "recon": rng.choice(["teno_d", "teno_d", "weno_ao", "weno_z", "teno5"]),
                "bc": rng.choice(["zerograd", "reflect", "periodic"]), "call": rng.choice(["advance", "step"])}
    if kind == "plane":
        top = 1400 if precision == "fp32" else 400
        tau = rng.choice(["euler", "euler", "ns", "zero"])
        return {"kind": kind, "nx": _log(rng, 24, top), "ny": _log(rng, 24, top), "precision": precision,
                "steps": rng.randint(1, 2), "tau": tau,
                "recon": rng.choice(["teno_d", "teno_d", "teno_d", "weno_ao", "weno_z", "teno5"]),
                "bc": "walls" if tau == "ns" else rng.choice(["zerograd", "periodic"]),
                "cfl": rng.choice([0.2, 0.5, 0.8]), "Pr": 0.73 if tau == "ns" else 1.0,
                "call": rng.choice(["advance", "step"])}
    if kind == "batch":
        return {"kind": kind, "count": _log(rng, 64, 1024), "nmin": rng.randint(100, 300),
                "nmax": rng.randint(400, 3000), "precision": precision,
                "steps": rng.randint(4, 16) if precision == "fp32" else rng.randint(1, 4)}
    top = 400 if precision == "fp32" else 128
    return {"kind": kind, "nx": _log(rng, 24, top), "ny": _log(rng, 24, top), "precision": precision,
            "steps": rng.randint(2, 6), "every": rng.randint(1, 4), "call": rng.choice(["object", "flow"])}


# ------------------------------------------------------------------ inputs
def _conserved(rho, u, v, p):
    E = p / (GAMMA - 1.0) + 0.5 * rho * (u * u + (0.0 if v is None else v * v))
    return torch.stack([rho, rho * u, E] if v is None else [rho, rho * u, rho * v, E]).contiguous()


def _waves(g, shape, amp, kmax):
    """A few seeded Fourier modes, periodic on the grid, at most about amp."""
    f = torch.zeros(shape, dtype=torch.float64, device="cuda")
    axes = [torch.arange(n, dtype=torch.float64, device="cuda").add_(0.5).div_(n) for n in shape]
    for _ in range(4):
        k = g.integers(1, kmax + 1, size=len(shape))
        ph, a = g.uniform(0, 2 * math.pi), amp * g.uniform(-0.5, 0.5)
        arg = sum(2 * math.pi * float(kk) * ax.reshape([-1 if i == j else 1 for j in range(len(shape))])
                  for i, (kk, ax) in enumerate(zip(k, axes)))
        f += a * torch.sin(arg + ph)
    return f


def _below(x, x0, n):
    """1 where x < x0, 0 beyond, over about eight of n cells: a jump as the
    scheme captures it, not the one-cell jump of a first step."""
    return 0.5 * (1 - torch.tanh((x - x0) * (0.25 * n)))


def _tube_state(g, nx):
    """A shock tube (Sod's states, jittered) over a density and pressure wave."""
    j = lambda s: 1.0 + s * g.uniform(-1, 1)  # noqa: E731
    left, right = (1.0 * j(0.1), 0.1 * g.uniform(-1, 1), 1.0 * j(0.1)), (0.125 * j(0.1), 0.0, 0.1 * j(0.1))
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) / nx
    at = _below(x, g.uniform(0.4, 0.6), nx)
    rho, u, p = (b + (a - b) * at for a, b in zip(left, right))
    kmax = max(1, min(8, nx // 32))
    return _conserved(rho * (1 + _waves(g, (nx,), 0.1, kmax)), u + _waves(g, (nx,), 0.05, kmax), None,
                      p * (1 + _waves(g, (nx,), 0.1, kmax)))[:, None, :].contiguous()


_QUADRANTS = [(1.0, -0.75, 0.5, 1.0), (3.0, -0.75, -0.5, 1.0), (1.0, -0.75, -0.5, 1.0), (2.0, 0.75, 0.5, 1.0)]


def _plane_state(g, nx, ny, viscous):
    """Riemann configuration 6 (or the viscous shock tube's two states) with
    jittered states and split, over waves in every field."""
    X = ((torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) / nx)[None, :]
    Y = ((torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny)[:, None]
    sx, sy = g.uniform(0.4, 0.8), g.uniform(0.4, 0.8)
    j = lambda v: v * (1.0 + 0.05 * g.uniform(-1, 1))  # noqa: E731
    kx = max(1, min(4, min(nx, ny) // 32))
    wave = lambda a: _waves(g, (ny, nx), a, kx)  # noqa: E731
    if viscous:
        states = [(120.0, 0.0, 0.0, 120.0 / GAMMA), (1.2, 0.0, 0.0, 1.2 / GAMMA)]
        f = [j(b) + (j(a) - j(b)) * _below(X, sx, nx) + 0 * Y for a, b in zip(*states)]
        return _conserved(f[0] * (1 + wave(0.05)), f[1] + wave(0.05), f[2] + wave(0.05), f[3] * (1 + wave(0.05)))
    q = [[j(v) for v in s] for s in _QUADRANTS]
    ax, ay = _below(X, sx, nx), _below(Y, sy, ny)
    f = [ay * (ax * q[0][k] + (1 - ax) * q[1][k]) + (1 - ay) * (ax * q[3][k] + (1 - ax) * q[2][k]) for k in range(4)]
    return _conserved(f[0] * (1 + wave(0.05)), f[1] + wave(0.05), f[2] + wave(0.05), f[3] * (1 + wave(0.05)))


def _smooth_state(g, nx, ny):
    """A smooth periodic flow: a diagonal wave of every field in a mean flow,
    24 to 48 cells long along each axis."""
    th = 0.0
    for n, shape in ((nx, (1, -1)), (ny, (-1, 1))):
        k = float(g.integers(-(-n // 48), max(1, n // 24) + 1))
        th = th + (2 * math.pi * k / n) * torch.arange(n, dtype=torch.float64, device="cuda").reshape(shape)
    w = lambda a: a * torch.sin(th + g.uniform(0, 2 * math.pi))  # noqa: E731
    return _conserved(1 + w(0.2), 1 + w(0.1), 0.7 + w(0.1), 1 + w(0.2))


def _batch_sizes(case):
    """The problems' cell counts: the case's, whatever the seed."""
    g = np.random.Generator(np.random.PCG64(2309))
    return g.integers(case["nmin"], case["nmax"] + 1, size=case["count"]).astype(np.int32)


def _batch_state(g, case):
    """(cells per problem, packed states): one Riemann problem each."""
    n = _batch_sizes(case)
    side = lambda: (np.exp(g.uniform(-0.4, 0.4, len(n))), g.uniform(-0.2, 0.2, len(n)), np.exp(g.uniform(-0.4, 0.4, len(n))))  # noqa: E731
    own = np.repeat(np.arange(len(n)), n)
    off = np.concatenate([[0], np.cumsum(n)[:-1]])
    x = torch.from_numpy((np.arange(int(n.sum())) - off[own] + 0.5) / n[own]).cuda()
    own = torch.from_numpy(own).cuda()
    pick = lambda v: torch.from_numpy(v).cuda()[own]  # noqa: E731
    at = _below(x, 0.5, torch.from_numpy(n.astype(np.float64)).cuda()[own])
    f = [pick(b) + pick(a - b) * at for a, b in zip(side(), side())]
    k = torch.from_numpy(g.integers(1, 5, len(n)).astype(np.float64)).cuda()[own]
    f[0] = f[0] * (1 + 0.05 * torch.sin(2 * math.pi * k * x))
    return n, _conserved(f[0], f[1], None, f[2])


_BC = {"zerograd": ("zerograd",) * 4, "periodic": ("periodic",) * 4, "reflect": ("reflect",) * 4,
       "walls": ("noslip", "noslip", "noslip", "symmetry")}
MU = 1.0 / 200.0


def _fixed_dt(W, h, cfl=0.4):
    """A stable time step for a call that takes one (cfl h / (|U| + a))."""
    return float(cfl / _rate(W, GAMMA, 0.0, h).max())


def prepare(case, seed):
    g = np.random.Generator(np.random.PCG64(int(seed)))
    kind, s = case["kind"], {"case": case}
    if kind == "batch":
        n, W = _batch_state(g, case)
        s.update(W=W, solver=gks.Batch(n, np.ones(len(n)), precision=case["precision"]))
        return s
    if kind == "noalloc":
        s["W"] = _tube_state(g, case["nx"])
        s.update(dt=_fixed_dt(s["W"], 1.0 / case["nx"]), out=torch.empty_like(s["W"]))
        return s
    if kind == "tube":
        s["W"] = _tube_state(g, case["nx"])
        s["solver"] = gks.Solver(1, case["nx"], bc=_BC[case["bc"]], precision=case["precision"], tau=case["tau"],
                                 recon=case["recon"])
    elif kind == "plane":
        s["W"] = _plane_state(g, case["nx"], case["ny"], case["bc"] == "walls")
        s["solver"] = gks.Solver(2, case["nx"], case["ny"], ly=0.5 if case["bc"] == "walls" else 1.0,
                                 bc=_BC[case["bc"]], precision=case["precision"], tau=case["tau"], cfl=case["cfl"],
                                 mu=MU if case["tau"] == "ns" else 0.0, Pr=case["Pr"], recon=case["recon"])
    else:
        s["W"] = _smooth_state(g, case["nx"], case["ny"])
        s["G"] = torch.stack([_waves(g, (case["ny"], case["nx"]), 1.0, 3) for _ in range(4)])
        s["solver"] = gks.Solver(2, case["nx"], case["ny"], bc=_BC["periodic"], precision=case["precision"], tau="zero")
        s["dt"] = _fixed_dt(s["W"], min(1.0 / case["nx"], 1.0 / case["ny"]))
        if case["call"] == "object":
            s["adjoint"] = gks.Adjoint(s["solver"], case["every"])
            s["adjoint"].reserve(case["steps"])
    s["out"] = torch.empty_like(s["W"])
    return s


def _typed(case, x):
    """A state in the type its path's digits are good for (see above)."""
    if case["precision"] == "fp64":
        return x
    return x.astype(np.float32) if isinstance(x, np.ndarray) else x.to(torch.float32)


def run(s):
    case = s["case"]
    kind, W = case["kind"], s["W"]
    if kind == "noalloc":
        gks.step1d_noalloc(W, s["out"], 1.0 / case["nx"], s["dt"], precision=case["precision"])
        return _typed(case, s["out"])
    S = s["solver"]
    if kind == "batch":
        S.set_state(W)
        S.advance_to(100.0, max_steps=case["steps"])
        return _typed(case, S.get_state())
    if kind == "adjoint" and case["call"] == "flow":
        W0 = W.detach().requires_grad_(True)
        WN = gks.flow(W0, S, case["steps"], s["dt"], case["every"])
        gW0, = torch.autograd.grad(WN, W0, s["G"])
        return _typed(case, WN.detach()), _typed(case, gW0)
    S.set_state(W)
    if kind == "adjoint":
        s["adjoint"].forward(case["steps"], s["dt"])
        WN = _typed(case, S.get_state(s["out"]))
        return WN, _typed(case, s["adjoint"].backward(s["G"]))
    if case["call"] == "advance":
        S.advance_to(100.0, max_steps=case["steps"])
    else:
        for _ in range(case["steps"]):
            S.step()
    return _typed(case, S.get_state(s["out"]))


# Arithmetic per cell of one stage in one direction, counted on the formulas
# with common parts formed once: a reconstruction about 75; the flux at a
# point about 300 (tau = 0), 500 (Euler), 600 (Navier-Stokes with Prandtl);
# the update 10 per variable.
def work(case):
    kind = case["kind"]
    if kind == "batch":
        n = float(_batch_sizes(case).sum())
        return {"bytes": 2 * 24 * n, "flops": n * case["steps"] * 2 * (3 * 75 + 400)}
    if kind in ("noalloc", "tube"):
        n = float(case["nx"])
        flux = 250 if case.get("tau") == "zero" else 400
        return {"bytes": 2 * 24 * n, "flops": n * case.get("steps", 1) * 2 * (3 * 75 + flux)}
    n = float(case["nx"] * case["ny"])
    flux = {"zero": 300, "euler": 500, "ns": 600}[case.get("tau", "zero")]
    step = 4 * (20 * 75 + 2 * flux + 40)
    if kind == "adjoint":  # forward, and the reverse of every operation (two products each)
        return {"bytes": 4 * 32 * n, "flops": 3 * n * case["steps"] * step}
    return {"bytes": 2 * 32 * n, "flops": n * case["steps"] * step}


# ------------------------------------------------------------------ 64-bit reference
def _coeffs(q):
    """Sub-stencil quadratics (b, c) and the quartic's Legendre-type u1..u4."""
    b = [(q[0] - 4 * q[1] + 3 * q[2]) / 2, (q[3] - q[1]) / 2, (-3 * q[2] + 4 * q[3] - q[4]) / 2]
    c = [(q[0] - 2 * q[1] + q[2]) / 2, (q[1] - 2 * q[2] + q[3]) / 2, (q[2] - 2 * q[3] + q[4]) / 2]
    u = [(11 * q[0] - 82 * q[1] + 82 * q[3] - 11 * q[4]) / 120, (-3 * q[0] + 40 * q[1] - 74 * q[2] + 40 * q[3] - 3 * q[4]) / 56,
         (-q[0] + 2 * q[1] - 2 * q[3] + q[4]) / 12, (q[0] - 4 * q[1] + 6 * q[2] - 4 * q[3] + q[4]) / 24]
    return b, c, u


def _weights(b, c, u, recon):
    """Weights of the quartic and the three quadratics in the reconstruction."""
    beta = [b[k] ** 2 + 13 / 3 * c[k] ** 2 for k in range(3)]
    beta.append((u[0] + u[2] / 10) ** 2 + 13 / 3 * (u[1] + 123 / 455 * u[3]) ** 2 + 781 / 20 * u[2] ** 2
                + 1421461 / 2275 * u[3] ** 2)
    if recon == "weno_ao":
        tau = ((beta[3] - beta[0]).abs() + (beta[3] - beta[1]).abs() + (beta[3] - beta[2]).abs()) / 3
        g = [(1 - D_HI) * (1 - D_LO) / 2, (1 - D_HI) * D_LO, (1 - D_HI) * (1 - D_LO) / 2, D_HI]
        om = [g[k] * (1 + (tau / (beta[k] + EPS_AO)) ** 2) for k in range(4)]
        tot = om[0] + om[1] + om[2] + om[3]
        w3 = om[3] / tot / D_HI
        return w3, [om[k] / tot - w3 * g[k] for k in range(3)]
    with torch.no_grad():  # the selection is piecewise constant
        t = [x + EPS for x in beta]
        m = torch.minimum(torch.minimum(t[0], t[1]), torch.minimum(t[2], t[3]))
        r = [(m / x) ** Q for x in t]
        small = r[0] + r[1] + r[2]
        large = (r[3] >= CT1 * (small + r[3])).to(m.dtype)
        keep = [(x >= CT2 * small).to(m.dtype) for x in r[:3]]
        n = (1 - large) / (keep[0] + keep[1] + keep[2])
        return large, [x * n for x in keep]


def _blend(q, xi, recon):
    """(value, xi-derivative) of the reconstruction at each point of xi."""
    b, c, u = _coeffs(q)
    w3, w = _weights(b, c, u, recon)
    ws = w[0] + w[1] + w[2]
    sb, sc = (w[0] * f[0] + w[1] * f[1] + w[2] * f[2] for f in (b, c))
    out = []
    for x in xi:
        p2, p3, p4 = x * x - 1 / 12, x ** 3 - 3 * x / 20, x ** 4 - 3 * x * x / 14 + 3 / 560
        d3, d4 = 3 * x * x - 3 / 20, 4 * x ** 3 - 3 * x / 7
        out.append(((w3 + ws) * q[2] + w3 * (u[0] * x + u[1] * p2 + u[2] * p3 + u[3] * p4) + sb * x + sc * p2,
                    w3 * (u[0] + 2 * u[1] * x + u[2] * d3 + u[3] * d4) + sb + 2 * sc * x))
    return out


def _mom(u, v, x2, x4, k, m):
    """<u^k v^m psi> of a unit-mass Maxwellian's tables, psi = (1, u, v, e)."""
    return [u[k] * v[m], u[k + 1] * v[m], u[k] * v[m + 1], 0.5 * (u[k + 2] * v[m] + u[k] * v[m + 2] + u[k] * v[m] * x2)]


def _mom_a(a, u, v, x2, x4, k, m):
    """<u^k v^m (a . psi) psi>."""
    M = lambda i, j: _mom(u, v, x2, x4, i, j)  # noqa: E731
    A, B, D, E, F = M(k, m), M(k + 1, m), M(k, m + 1), M(k + 2, m), M(k, m + 2)
    xi = [x2 * A[0], x2 * A[1], x2 * A[2], 0.5 * (x2 * (u[k + 2] * v[m] + u[k] * v[m + 2]) + x4 * u[k] * v[m])]
    return [a[0] * A[i] + a[1] * B[i] + a[2] * D[i] + 0.5 * a[3] * (E[i] + F[i] + xi[i]) for i in range(4)]


def _tables(U, V, T, dim, half=0):
    """<u^n> (half: over u > 0 or u < 0) and <v^n>, n = 0..6."""
    if half:
        z = U / torch.sqrt(2 * T)
        u = [0.5 * torch.erfc(-half * z)]
        u.append(U * u[0] + half * torch.exp(-z * z) * torch.sqrt(T / (2 * math.pi)))
    else:
        u = [torch.ones_like(U), U]
    for n in range(5):
        u.append(U * u[n + 1] + (n + 1) * T * u[n])
    if dim == 1:
        return u, [torch.ones_like(U)] + [torch.zeros_like(U)] * 6
    v = [torch.ones_like(V), V]
    for n in range(5):
        v.append(V * v[n + 1] + (n + 1) * T * v[n])
    return u, v


def _slope(d, rho, U, V, T, K, dim):
    """a with <a . psi> = d / rho (the Maxwellian's linear system in closed form)."""
    b = [x / rho for x in d]
    n = K + dim
    E = 0.5 * (U * U + V * V + n * T)
    r1, r2, r3 = b[1] - U * b[0], b[2] - V * b[0], 2 * (b[3] - E * b[0])
    a3 = (r3 - 2 * U * r1 - 2 * V * r2) / (n * T * T)
    a2 = r2 / T - V * a3 if dim == 2 else torch.zeros_like(U)
    a1 = r1 / T - U * a3
    return [b[0] - U * a1 - V * a2 - E * a3, a1, a2, a3]


def _phi(x):
    """The six time integrals of the BGK solution over [0, x] in units of tau."""
    e = torch.expm1(-x)
    full = [x + e, -2 * x - (x + 2) * e, x * x / 2 - x - e, -e, x + (x + 2) * e, e]
    ser = [torch.zeros_like(x) for _ in range(6)]
    y, f = torch.where(x < 0.5, x, torch.zeros_like(x)), 1.0
    for n in range(1, 17):
        f *= -1.0 / n
        t = f * y ** n
        ser[3] = ser[3] - t
        ser[5] = ser[5] + t
        ser[4] = ser[4] + (2 - n) * t
        if n >= 2:
            ser[0] = ser[0] + t
        if n >= 3:
            ser[1] = ser[1] + (n - 2) * t
            ser[2] = ser[2] - t
    return [torch.where(x < 0.5, s, g) for s, g in zip(ser, full)]


def _pressure(W):
    return (GAMMA - 1) * (W[3] - 0.5 * (W[1] ** 2 + W[2] ** 2) / W[0])


def _flux(L, R, dt, dim, tau, mu, Pr):
    """(F, dF/dt) of the two sides' (W, Wn, Wt) in the face's frame."""
    K = (5 - 3 * GAMMA) / (GAMMA - 1) + 1 if dim == 2 else (3 - GAMMA) / (GAMMA - 1)
    add = lambda x, y: [a + b for a, b in zip(x, y)]  # noqa: E731
    W0, Wn, Wt, S3, S4, S5, N4, N5 = ([0.0] * 4 for _ in range(8))
    p = []
    for (W, Dn, Dt), half in ((L, 1), (R, -1)):
        rho, U, V = W[0], W[1] / W[0], W[2] / W[0]
        p.append(_pressure(W))
        T = p[-1] / rho
        x2, x4 = K * T, K * (K + 2) * T * T
        u, v = _tables(U, V, T, dim, half)
        an, at = _slope(Dn, rho, U, V, T, K, dim), _slope(Dt, rho, U, V, T, K, dim)
        mom = lambda k, m: [rho * y for y in _mom(u, v, x2, x4, k, m)]  # noqa: E731
        mom_a = lambda a, k, m: [rho * y for y in _mom_a(a, u, v, x2, x4, k, m)]  # noqa: E731
        W0, Wn, Wt = add(W0, mom(0, 0)), add(Wn, mom_a(an, 0, 0)), add(Wt, mom_a(at, 0, 0))
        if tau == "zero":
            continue
        uf, vf = _tables(U, V, T, dim)
        A = _slope([-(x + y) for x, y in zip(_mom_a(an, uf, vf, x2, x4, 1, 0), _mom_a(at, uf, vf, x2, x4, 0, 1))],
                   1.0, U, V, T, K, dim)
        S3, S5 = add(S3, mom(1, 0)), add(S5, mom_a(A, 1, 0))
        S4 = add(S4, add(mom_a(an, 2, 0), mom_a(at, 1, 1)))
        N5, N4 = add(N5, mom_a(A, 0, 0)), add(N4, add(mom_a(an, 1, 0), mom_a(at, 0, 1)))
    rho, U, V = W0[0], W0[1] / W0[0], W0[2] / W0[0]
    p0 = _pressure(W0)
    T = p0 / rho
    x2, x4 = K * T, K * (K + 2) * T * T
    u, v = _tables(U, V, T, dim)
    an, at = _slope(Wn, rho, U, V, T, K, dim), _slope(Wt, rho, U, V, T, K, dim)
    m_a = lambda a, k, m: [rho * y for y in _mom_a(a, u, v, x2, x4, k, m)]  # noqa: E731
    Wtime = [-(x + y) for x, y in zip(m_a(an, 1, 0), m_a(at, 0, 1))]
    A = _slope(Wtime, rho, U, V, T, K, dim)
    F0, F2 = [rho * y for y in _mom(u, v, x2, x4, 1, 0)], m_a(A, 1, 0)
    if tau == "zero":
        return F0, F2
    F1 = add(m_a(an, 2, 0), m_a(at, 1, 1))
    jump = (p[0] - p[1]).abs() / (p[0] + p[1])
    tc = (C1 + C2 * jump) * dt if tau == "euler" else mu / p0 + C2 * jump * dt
    full, half = _phi(dt / tc), _phi(0.5 * dt / tc)
    pw = [1, 2, 2, 1, 2, 2]
    qF = [(4 * h - f) * tc ** k / dt for f, h, k in zip(full, half, pw)]
    qD = [4 * (f - 2 * h) * tc ** k / dt ** 2 for f, h, k in zip(full, half, pw)]

    def total(q, terms):
        return [sum(c * t[i] for c, t in zip(q, terms)) for i in range(4)]

    F, dF = (total(q, (F0, F1, F2, S3, S4, S5)) for q in (qF, qD))
    if tau == "ns" and Pr != 1.0:  # heat flux (relative to U0, V0) scaled by 1/Pr
        dens = ([rho * torch.ones_like(U), rho * U, rho * V, W0[3]], [-x for x in Wtime], Wtime, W0, N4, N5)
        ke = 0.5 * (U * U + V * V)
        for f, q in ((F, qF), (dF, qD)):
            M = total(q, dens)
            f[3] = f[3] + (1 / Pr - 1) * (f[3] - U * f[1] - V * f[2] + (ke + U * U) * f[0] + U * V * M[2] - U * M[3]
                                          - U * ke * M[0])
    return F, dF


def _ok(W):
    return (W[0] > 0) & (_pressure(W) > 0)


def _safe(W, Dn, Dt, cell):
    """A non-physical point takes the adjacent cell's average and no slopes."""
    ok = _ok(W)
    if bool(ok.all()):
        return W, Dn, Dt
    z = torch.zeros_like(W[0])
    return ([torch.where(ok, a, b) for a, b in zip(W, cell)], [torch.where(ok, a, z) for a in Dn],
            [torch.where(ok, a, z) for a in Dt])


def _divergence(W, h, ht, dt, dim, tau, mu, Pr, recon):
    """The stage's flux differences along the last axis: (of F, of dF), from a
    state [4][rows][cells] in the face's frame with three ghosts on each side
    (1-D: one row without ghosts)."""
    n = W.shape[-1] - 4
    q = [W[..., s:s + n] for s in range(5)]
    (vp, dp), (vm, dm) = _blend(q, (0.5, -0.5), recon)
    sides = [(vp[..., :-1], dp[..., :-1] / h), (vm[..., 1:], dm[..., 1:] / h)]
    if dim == 1:
        cells = [W[..., 2:-3], W[..., 3:-2]]
        pts = [[(list(v), list(d), [torch.zeros_like(v[0])] * 4) for v, d in sides]]
    else:
        m = W.shape[1] - 6
        cells = [W[:, 3:-3, 2:-3], W[:, 3:-3, 3:-2]]
        xi = (-0.5 / math.sqrt(3), 0.5 / math.sqrt(3))
        both = []
        for v, d in sides:
            val = _blend([v[:, 1 + s:1 + s + m] for s in range(5)], xi, recon)
            slp = _blend([d[:, 1 + s:1 + s + m] for s in range(5)], xi, recon)
            both.append([(list(a), list(c), list(b / ht)) for (a, b), (c, _) in zip(val, slp)])
        pts = list(zip(*both))
    F = dF = None
    for L, R in pts:
        f, d = _flux(_safe(*L, list(cells[0])), _safe(*R, list(cells[1])), dt, dim, tau, mu, Pr)
        f, d = torch.stack(f) / len(pts), torch.stack(d) / len(pts)
        F, dF = (f, d) if F is None else (F + f, dF + d)
    return F[..., 1:] - F[..., :-1], dF[..., 1:] - dF[..., :-1]


_FLIP = {"symmetry": (1,), "reflect": (1,), "noslip": (1, 2)}


def _ghost(W, axis, lo, hi):
    """Three ghosts on both sides along `axis` (of 4 slots; normal slot 1)."""
    n = W.shape[axis]
    take = lambda i: W.index_select(axis, torch.tensor(i, device=W.device))  # noqa: E731
    if lo == "periodic":
        return torch.cat([take([n - 3, n - 2, n - 1]), W, take([0, 1, 2])], axis)

    def side(bc, edge, mirror):
        if bc == "zerograd":
            return take([edge] * 3)
        g = take(mirror)
        sign = torch.ones(4, dtype=W.dtype, device=W.device)
        sign[list(_FLIP[bc])] = -1.0
        return g * sign.reshape(4, *[1] * (W.dim() - 1))

    return torch.cat([side(lo, 0, [2, 1, 0]), W, side(hi, n - 1, [n - 1, n - 2, n - 3])], axis)


def _swap(W):
    """x and y exchanged: momentum slots and axes."""
    return torch.stack([W[0], W[2], W[1], W[3]]).transpose(1, 2)


def _stage_div(W, hx, hy, dt, dim, bc, tau, mu, Pr, recon):
    """Flux differences over h of both directions."""
    args = (dt, dim, tau, mu, Pr, recon)
    if dim == 1:
        f, d = _divergence(_ghost(W, 2, bc[0], bc[1]), hx, 1.0, *args)
        return f / hx, d / hx
    # x ghosts first, then y ghosts over the full width
    G = _swap(_ghost(_swap(_ghost(W, 2, bc[0], bc[1])), 2, bc[2], bc[3]))
    f, d = _divergence(G, hx, hy, *args)
    f2, d2 = _divergence(_swap(G), hy, hx, *args)
    return f / hx + _swap(f2) / hy, d / hx + _swap(d2) / hy


def _step(W, dt, div):
    """One two-stage fourth-order step; div(W) gives the flux differences."""
    F, dF = div(W)
    _, dS = div(W - dt * (F / 2 + dt / 8 * dF))
    return W - dt * (F + dt / 6 * dF) - dt * (dt / 3 * dS)


def _rate(W, gamma, mu, h):
    rho, q = W[0], (W[1:-1] ** 2).sum(0)
    a = torch.sqrt(gamma * (gamma - 1) * (W[-1] - 0.5 * q / rho) / rho)
    s = (torch.sqrt(q) / rho + a) / h
    return torch.maximum(s, 4 * mu / rho / (h * h)) if mu > 0 else s


def _four(W):
    """1-D states in four slots (no tangential momentum)."""
    return torch.stack([W[0], W[1], torch.zeros_like(W[0]), W[2]])


def _three(W):
    return torch.stack([W[0], W[1], W[3]])


def _exact_batch(case, g):
    n, W = _batch_state(g, case)
    n = torch.from_numpy(n.astype(np.int64)).cuda()
    own = torch.repeat_interleave(torch.arange(len(n), device="cuda"), n)
    off = torch.cumsum(n, 0) - n
    # every problem's cells with three copies of its end cells on both sides
    ng = n + 6
    owng = torch.repeat_interleave(torch.arange(len(n), device="cuda"), ng)
    offg = torch.cumsum(ng, 0) - ng
    at = torch.arange(len(owng), device="cuda") - offg[owng] - 3
    src = off[owng] + torch.minimum(at.clamp(min=0), n[owng] - 1)
    face = torch.arange(len(own), device="cuda") - off[own] + offg[own] + 3  # a cell's place among the ghosted
    h = 1.0 / n.to(torch.float64)
    hg, hc = h[owng], h[own]
    W = _four(W)[:, None, :]
    for _ in range(case["steps"]):
        sig = torch.zeros(len(n), dtype=torch.float64, device="cuda")
        sig = sig.scatter_reduce(0, own, _rate(_three(W)[:, 0], GAMMA, 0.0, hc), "amax")
        dtp = 0.5 / sig

        def div(S):
            # faces of the whole ghosted row: cell c's low face is window c - 3
            f, d = _divergence(S[:, :, src], hg[2:-3], 1.0, dtp[owng][2:-3], 1, "euler", 0.0, 1.0, "teno_d")
            return f[..., face - 3] / hc, d[..., face - 3] / hc

        W = _step(W, dtp[own], div)
    return _three(W)[:, 0]


def exact(case, seed):
    """The scheme on the same inputs in float64 (None: WENO5-Z and TENO5)."""
    g = np.random.Generator(np.random.PCG64(int(seed)))
    kind = case["kind"]
    if kind == "batch":
        with torch.no_grad():
            return _exact_batch(case, g).cpu().numpy()
    recon = case.get("recon", "teno_d")
    if recon not in ("teno_d", "weno_ao"):
        return None
    dim = 1 if kind in ("noalloc", "tube") else 2
    if dim == 1:
        W = _four(_tube_state(g, case["nx"]))
        bc, hx, hy = _BC[case.get("bc", "zerograd")], 1.0 / case["nx"], 1.0
    elif kind == "plane":
        walls = case["bc"] == "walls"
        W = _plane_state(g, case["nx"], case["ny"], walls)
        bc, hx, hy = _BC[case["bc"]], 1.0 / case["nx"], (0.5 if walls else 1.0) / case["ny"]
    else:
        W = _smooth_state(g, case["nx"], case["ny"])
        G = torch.stack([_waves(g, (case["ny"], case["nx"]), 1.0, 3) for _ in range(4)])
        bc, hx, hy = _BC["periodic"], 1.0 / case["nx"], 1.0 / case["ny"]
    h = hx if dim == 1 else min(hx, hy)
    tau, Pr = case.get("tau", "zero" if kind == "adjoint" else "euler"), case.get("Pr", 1.0)
    mu = MU if tau == "ns" else 0.0
    step = lambda S, dt: _step(S, dt, lambda X: _stage_div(X, hx, hy, dt, dim, bc, tau, mu, Pr, recon))  # noqa: E731
    if kind == "adjoint":
        dt, states = _fixed_dt(W, h), [W]
        with torch.no_grad():
            for _ in range(case["steps"]):
                states.append(step(states[-1], dt))
        for S in reversed(states[:-1]):
            S = S.detach().requires_grad_(True)
            G, = torch.autograd.grad(step(S, dt), S, G)
        return states[-1], G
    with torch.no_grad():
        for _ in range(case.get("steps", 1)):
            dt = _fixed_dt(_three(W) if dim == 1 else W, h) if kind == "noalloc" else \
                float(case.get("cfl", 0.5) / _rate(_three(W) if dim == 1 else W, GAMMA, mu, h).max())
            W = step(W, dt)
    return _three(W) if dim == 1 else W
