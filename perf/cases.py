"""What the solver is used for, as cases that can be timed and compared.

A case is one pass of a user's program through the public entry points: load an
initial state, advance it, read the result.  The sizes are those of the
repository's workloads (the paper's Sec. 5 problems, the ensemble, the batch of
lines, the adjoint window) and of its tests.

Kinds: "grid" (Solver, fixed time steps or a CFL step each step, device or
pinned host arrays), "ensemble" (Ensemble), "lines" (Lines), "adjoint"
(Solver.vjp_steps).

An FP64 run's state is returned as it is.  A mixed-precision run's results
carry FP32 accuracy (its interface values are FP32, an averaged gradient is a
difference of two of them over h): its state is kept as one float32 array of
the values and their increments over a node's interval, h times the averaged
gradients.

exact() is the scheme in plain torch operations in 64 bits: moments from
tables, slopes from the moment system's closed form, whole fields at once; the
adjoint is torch.autograd through it.
"""
import math

import numpy as np
import torch

from paper_2606_17772_gb300 import fdcgks, inputs

PREC = {"fp64": fdcgks.FP64, "mixed": fdcgks.MIXED}


def listed():
    return [
        # config 2's largest grid, the benchmark's workload, in both precisions: a time loop with a known step
        dict(name="vortex_fp64_1024", kind="grid", problem="vortex", precision="fp64", nx=1024, ny=1024, steps=2,
             loop="fixed", io="device"),
        dict(name="vortex_mixed_1024", kind="grid", problem="vortex", precision="mixed", nx=1024, ny=1024, steps=10,
             loop="fixed", io="device"),
        # config 2's smallest grid, FP64, a CFL step each step as runs.advance takes them
        dict(name="vortex_fp64_128", kind="grid", problem="vortex", precision="fp64", nx=128, ny=128, steps=10,
             loop="cfl", io="device"),
        # the smallest grid of the sweeps, odd, mixed: launches and the host round trip of the CFL step count
        dict(name="vortex_mixed_33", kind="grid", problem="vortex", precision="mixed", nx=33, ny=33, steps=20,
             loop="cfl", io="device"),
        # config 3 at its size: no-slip walls, viscosity, symmetry, strong jump, a CFL step each step
        dict(name="tube_mixed_1000x500", kind="grid", problem="tube", precision="mixed", nx=1000, ny=500, steps=4,
             loop="cfl", io="device"),
        # the same walls on a coarse odd grid in FP64 (a resolution study's first grid)
        dict(name="tube_fp64_251x125", kind="grid", problem="tube", precision="fp64", nx=251, ny=125, steps=3,
             loop="cfl", io="device"),
        # the paper's double Mach grid: characteristic reconstruction, 6-2 flux, split and moving sides
        dict(name="double_mach_fp64_960x240", kind="grid", problem="double_mach", precision="fp64", nx=960, ny=240,
             steps=2, loop="cfl", io="device"),
        # a program that keeps its state in pinned host memory between calls
        dict(name="host_fp64_512", kind="grid", problem="vortex", precision="fp64", nx=512, ny=512, steps=1,
             loop="fixed", io="host"),
        # config 4 with fewer members: uneven vortices, each with its own CFL step
        dict(name="ensemble_mixed_40", kind="ensemble", precision="mixed", members=40, nmin=32, nmax=512, steps=4),
        # config 1: one Sod line with the one-dimensional scheme, its own CFL steps, one launch (its first 20
        # steps: later the scheme itself turns rounding into visible differences behind the shock)
        dict(name="sod_line_fp64_200", kind="lines", problem="sod", precision="fp64", n=200, batch=1, loop="run",
             t_end=0.015),
        # a batch of blast-wave lines that fills the GPU, fixed steps
        dict(name="blast_lines_fp64_608x400", kind="lines", problem="blast", precision="fp64", n=400, batch=608,
             loop="fixed", steps=10),
        # config 5's grid: gradient through a window of steps, the variant that differences can check
        dict(name="adjoint_fp64_256", kind="adjoint", precision="fp64", nx=256, steps=4, checkpoint=2),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "ensemble", "lines", "lines", "adjoint"])
    precision = rng.choice(["fp64", "mixed"])
    if kind == "grid":
        problem = rng.choice(["vortex", "vortex", "tube", "double_mach"])
        nx = _log(rng, {"vortex": 32, "tube": 200, "double_mach": 480}[problem], 1000 if precision == "mixed" else 700)
        ny = {"vortex": nx, "tube": max(16, nx // 2), "double_mach": max(16, nx // 4)}[problem]
        steps = rng.randint(1, 8) if nx < 400 else rng.randint(1, 3)
        if problem == "tube":
            steps = min(steps, 4)
        if problem == "double_mach":
            steps = 1 if precision == "mixed" else min(steps, 2)
        return dict(kind="grid", problem=problem, precision=precision, nx=nx, ny=ny, steps=steps,
                    loop=rng.choice(["fixed", "cfl"]), io=rng.choice(["device", "device", "host"]))
    if kind == "ensemble":
        return dict(kind="ensemble", precision=precision, members=_log(rng, 2, 24), nmin=32,
                    nmax=_log(rng, 48, 300), steps=rng.randint(1, 4))
    if kind == "lines":
        if rng.random() < 0.5:
            n = _log(rng, 20, 300)
            return dict(kind="lines", problem="sod", precision=precision, n=n, batch=1, loop="run",
                        t_end=rng.uniform(1.0, 3.0) / n)
        return dict(kind="lines", problem="blast", precision=precision, n=_log(rng, 64, 600),
                    batch=_log(rng, 1, 400), loop="fixed", steps=rng.randint(2, 10))
    return dict(kind="adjoint", precision="fp64", nx=_log(rng, 32, 256), steps=rng.randint(1, 4),
                checkpoint=rng.randint(1, 3))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _ripple(c, rng, amp):
    """The problem's initial data with seeded smooth ripples of density and pressure."""
    base, Lx, Ly = c.prim, c.x1 - c.x0, c.y1 - c.y0
    k = rng.integers(1, 4, size=(2, 2, 2))
    a = rng.uniform(0.3, 1.0, size=(2, 2)) * amp
    ph = rng.uniform(0.0, 2.0 * math.pi, size=(2, 2))

    def wave(v, x, y):
        f = 1.0
        for m in range(2):
            yy = (y - c.y0) / Ly * k[v, m, 1] if c.ny > 1 else 0.0
            f = f + a[v, m] * np.cos(2 * math.pi * (k[v, m, 0] * (x - c.x0) / Lx + yy) + ph[v, m])
        return f

    def prim(x, y):
        rho, U, V, p = base(x, y)
        return rho * wave(0, x, y), U, V, p * wave(1, x, y)
    c.prim = prim
    return c


def _scaled(c, rng):
    """A shock tube with seeded left and right states around the problem's own."""
    base, a = c.prim, rng.uniform(0.95, 1.05, size=4)

    def prim(x, y):
        rho, U, V, p = base(x, y)
        left = x < 0.5
        return rho * np.where(left, a[0], a[1]), U, V, p * np.where(left, a[2], a[3])
    c.prim = prim
    return c


def _problem(case, seed):
    """(inputs.Case, CFL number, fixed time step) of a grid or adjoint case."""
    rng = np.random.default_rng(seed)
    name, nx = case.get("problem", "vortex"), case["nx"]
    if name == "vortex":
        kw = dict(geno_variant=2, tau_c1=0.05, tau_c2=0.0) if case["kind"] == "adjoint" else {}
        c = inputs.vortex(nx, strength=rng.uniform(1.0, 5.0), xc=rng.uniform(0, 10), yc=rng.uniform(0, 10), **kw)
        return c, 0.2, 0.2 * c.hx / 3.2
    if name == "tube":
        c = _ripple(inputs.viscous_shock_tube(nx, case["ny"], geno_variant=1, tau_c2=25.0), rng, 0.01)
        return c, 0.4, min(0.4 * c.hy / 1.2, 0.4 * c.hy * c.hy / (8.0 * 0.005 / 1.1)) * 0.9
    c = _ripple(inputs.double_mach(nx, case["ny"], flux_variant=62, recon_vars=1), rng, 0.002)
    return c, 0.4, 0.4 * c.hx / 14.0


def _line_problem(case, seed):
    rng = np.random.default_rng(seed)
    B, n = case["batch"], case["n"]
    W, X = [], []
    base = None
    for b in range(min(B, 8)):   # eight different lines; a larger batch repeats them, scaled
        if case["problem"] == "sod":
            c = _scaled(inputs.sod_strip(n, 1, geno_variant=1), rng)
        else:
            c = _ripple(inputs.woodward_colella(n, flux_variant=62, geno_variant=1), rng, 0.01)
        base = base or c
        w, x = inputs.line_state(c)
        W.append(w)
        X.append(x)
    s = rng.uniform(0.9, 1.1, size=(B, 1, 1))   # density, momentum and energy scaled together: the same speeds
    W = np.ascontiguousarray(np.stack([W[b % len(W)] for b in range(B)]) * s)
    X = np.ascontiguousarray(np.stack([X[b % len(X)] for b in range(B)]) * s)
    return base, W, X, 0.3, 2e-5 * 400.0 / n


def _members(case, seed):
    """Vortices on uneven grids (the sizes the case's own, log-spaced), strengths and centres seeded."""
    rng, M = np.random.default_rng(seed), case["members"]
    ratio = case["nmax"] / case["nmin"]
    n = [int(round(case["nmin"] * ratio ** ((k * 7 % M) / max(1, M - 1)))) for k in range(M)]
    return [inputs.vortex(k, strength=rng.uniform(1.0, 5.0), xc=rng.uniform(0, 10), yc=rng.uniform(0, 10)) for k in n]


def _dev(arrs):
    return [torch.from_numpy(a).cuda() for a in arrs]


def _misfit(c, seed):
    """dJ/d(final state) of the adjoint window: a density residual on the primary grid."""
    rng = np.random.default_rng([seed, 1])
    X, Y = c.node_xy(False)
    bump = np.zeros_like(X)
    for _ in range(8):
        cx, cy = rng.uniform(0, 10, 2)
        bump += rng.uniform(-1e-3, 1e-3) * np.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / 0.5)
    return bump * c.hx * c.hy


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        ms = _members(case, seed)
        e = fdcgks.Ensemble.from_cases(ms, PREC[case["precision"]])
        S = [_dev(m.initial_state()) for m in ms]
        return dict(case=case, e=e, S=S, out=[[torch.empty_like(t) for t in s] for s in S], h=[(m.hx, m.hy) for m in ms])
    if kind == "lines":
        c, W, X, cfl, dt = _line_problem(case, seed)
        L = fdcgks.Lines.from_case(c, case["batch"], precision=PREC[case["precision"]])
        return dict(case=case, L=L, S=_dev((W, X)), cfl=cfl, dt=dt, h=c.hx)
    c, cfl, dt = _problem(case, seed)
    s = fdcgks.Solver.from_case(c, PREC[case["precision"]])
    S = c.initial_state()
    if kind == "adjoint":
        S = _dev(S)
        a = [torch.zeros_like(t) for t in S]
        a[0][0] = torch.from_numpy(_misfit(c, seed)).cuda()
        return dict(case=case, s=s, S=S, a=a, dt=dt)
    if case["io"] == "host":
        S = [torch.from_numpy(a).pin_memory() for a in S]
        out = [torch.empty(t.shape, dtype=torch.float64).pin_memory() for t in S]
    else:
        S = _dev(S)
        out = [torch.empty_like(t) for t in S]
    return dict(case=case, s=s, S=S, out=out, cfl=cfl, dt=dt, h=(c.hx, c.hy))


def _snapshot(case, arrs, h, dtype=torch.float32):
    """The state as a program keeps it (grid: W, G of both grids; lines: W, W_x)."""
    if case["precision"] == "fp64":
        return list(arrs)
    if len(arrs) == 2:
        return [torch.cat([arrs[0], arrs[1] * h], dim=1).to(dtype)]
    return [torch.cat([W, G[0] * h[0], G[1] * h[1]]).to(dtype) for W, G in (arrs[:2], arrs[2:])]


def _times(case, t):
    return t if case["precision"] == "fp64" else t.astype(np.float32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "grid":
        s = state["s"]
        s.set_state(*state["S"])
        if case["loop"] == "fixed":
            s.steps(state["dt"], case["steps"])
        else:
            for _ in range(case["steps"]):
                s.step(s.cfl_dt(state["cfl"]))
        return _snapshot(case, s.get_state(out=state["out"]), state["h"])
    if kind == "ensemble":
        e = state["e"]
        for m, S in enumerate(state["S"]):
            e.set_state(m, *S)
        e.run(case["steps"], cfl=0.2)
        out = [_snapshot(case, e.get_state(m, out=o), h) for m, (o, h) in enumerate(zip(state["out"], state["h"]))]
        t, _, status = e.status()
        return [torch.cat([x.reshape(-1) for o in out for x in o]), _times(case, t), status]
    if kind == "lines":
        L = state["L"]
        L.set_state(*state["S"])
        if case["loop"] == "run":
            t, k = L.run(case["t_end"], cfl=state["cfl"])
            return _snapshot(case, L.get_state(), state["h"]) + [k]
        L.steps(state["dt"], case["steps"])
        return _snapshot(case, L.get_state(), state["h"])
    return list(state["s"].vjp_steps(state["dt"], case["steps"], state["S"], state["a"],
                                     checkpoint_every=case["checkpoint"]))


def work(case):
    """Bytes: the state read and the result written, 12 FP64 values a node each way.  Flops: what a step's
    arithmetic takes with moments in closed form (per node and stage two half-point line reconstructions of 4
    components, two interface solves, 8 node derivatives and a nodal flux, the compact update)."""
    step = 6.5e3
    if case["kind"] == "lines":
        n = case["n"] * case["batch"]
        k = case["steps"] if case["loop"] == "fixed" else case["t_end"] / (0.3 / (2.2 * case["n"]))
        return {"bytes": n * 6 * 16.0, "flops": 2.4e3 * n * k}
    if case["kind"] == "ensemble":
        a, b = math.log(case["nmin"]), math.log(case["nmax"])
        n2 = (math.exp(2 * b) - math.exp(2 * a)) / (2 * (b - a))   # mean of n^2, log-uniform n
        nodes = 2.0 * n2 * case["members"]
        return {"bytes": nodes * 12 * 16.0, "flops": step * nodes * case["steps"]}
    nodes = 2.0 * case["nx"] * case.get("ny", case["nx"])
    if case["kind"] == "adjoint":
        return {"bytes": nodes * 12 * 24.0, "flops": 4 * step * nodes * case["steps"]}
    return {"bytes": nodes * 12 * 16.0, "flops": step * nodes * case["steps"]}


# ---------------------------------------------------------------------------
# the scheme in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _geno(var, I0, I1, I2, d):
    r, eps = (3, 1e-15) if var == 1 else (2, 1e-12)
    lo, hi = torch.minimum(I0, torch.minimum(I1, I2)), torch.maximum(I0, torch.maximum(I1, I2))
    tau = (0.5 * (I1 + I2) - I0).abs()
    aH, aL = 1 + (tau / (hi + eps)) ** r, 1 + (tau / (lo + eps)) ** r
    chi = torch.tanh(40.0 * aH / (aH + aL)) / math.tanh(20.0)
    w = [dk / (I + 1e-6) ** 2 for dk, I in zip(d, (I0, I1, I2))]
    s = w[0] + w[1] + w[2]
    return chi, [x / s for x in w]


def _left(var, Q, X, h):
    """Value, derivative and path function at the middle of four nodes, from the left (App. C1)."""
    PH = (7 * Q[0] + 35 * Q[1] + 21 * Q[2] + Q[3] + (X[0] + 22 * X[1] - 7 * X[2]) * h) / 64
    PD = -((Q[0] + 45 * Q[1] - 45 * Q[2] - Q[3]) / h + 9 * (X[1] + X[2])) / 30
    if var == 2:
        return PH, PD, torch.ones_like(PH)
    c, b = 13.0 / 12.0, Q[1] - Q[0]
    I0 = 4 * c * (b - X[0] * h) ** 2 + (2 * b - X[0] * h) ** 2
    I1 = c * (Q[0] - 2 * Q[1] + Q[2]) ** 2 + (Q[2] - Q[0]) ** 2 / 4
    I2 = c * (Q[1] - 2 * Q[2] + Q[3]) ** 2 + (3 * Q[1] - 4 * Q[2] + Q[3]) ** 2 / 4
    chi, w = _geno(var, I0, I1, I2, (1, 8, 1) if var == 1 else (8, 1, 1))
    q = ((-5 * Q[0] + 9 * Q[1] - 3 * X[0] * h) / 4, (-Q[0] + 6 * Q[1] + 3 * Q[2]) / 8, (3 * Q[1] + 6 * Q[2] - Q[3]) / 8)
    D = (Q[2] - Q[1]) / h
    L = w[0] * q[0] + w[1] * q[1] + w[2] * q[2]
    LD = w[0] * (3 * b / h - 2 * X[0]) + (w[1] + w[2]) * D
    return chi * PH + (1 - chi) * L, chi * PD + (1 - chi) * LD, chi


def _both(var, Q, X, h):
    """Left and right states: the right one is the mirror image of the left."""
    vl, dl, cl = _left(var, Q, X, h)
    vr, dr, cr = _left(var, Q[::-1], [-x for x in X[::-1]], h)
    return vl, dl, vr, -dr, cl, cr


def _node_derivative(var, Q, X, h):
    PD = (9 * (Q[0] - Q[2]) / h + X[0] + 46 * X[1] + X[2]) / 30
    if var == 2:
        return PD
    c, a, b = 13.0 / 12.0, Q[1] - Q[0], Q[2] - Q[1]
    I0 = c * (Q[0] - 2 * Q[1] + Q[2]) ** 2 + (Q[2] - Q[0]) ** 2 / 4
    I1 = 4 * c * (a - X[0] * h) ** 2 + (2 * a - X[0] * h) ** 2
    I2 = 4 * c * (b - X[2] * h) ** 2 + (2 * b - X[2] * h) ** 2
    chi, w = _geno(var, I0, I1, I2, (8, 1, 1))
    LD = w[0] * (Q[2] - Q[0]) / (2 * h) + w[1] * (2 * a / h - X[0]) + w[2] * (2 * b / h - X[2])
    return chi * PD + (1 - chi) * LD


def _safe(v, d, chi, node):
    """A state without positive density and pressure is replaced by its node's, with no slope and chi 0."""
    ok = (v[0] > 0) & (2 * v[3] * v[0] > v[1] ** 2 + v[2] ** 2)
    return torch.where(ok, v, node), torch.where(ok, d, torch.zeros_like(d)), torch.where(ok, chi, torch.zeros_like(chi))


def _line(c, Q, X, h, normal):
    """States at the middle of a four-node line: Q, X lists of 4 tensors [4, ...] (conservative)."""
    if not c.recon_vars:
        vl, dl, vr, dr, cl, cr = _both(c.geno_variant, Q, X, h)
        chi = torch.minimum(cl[0], cr[0])
    else:
        n, t = (1, 2) if normal == 0 else (2, 1)
        r, mn, mt, E = (0.5 * (Q[1] + Q[2])[[0, n, t, 3]]).unbind(0)
        g1 = c.gamma - 1
        u, v = mn / r, mt / r
        q2 = u * u + v * v
        p = g1 * (E - 0.5 * r * q2)
        a, H = torch.sqrt(c.gamma * p / r), (E + p) / r
        b1, b2, z, o = g1 / a ** 2, 0.5 * g1 / a ** 2 * q2, torch.zeros_like(u), torch.ones_like(u)
        Lm = [[(b2 + u / a) / 2, -(b1 * u + 1 / a) / 2, -b1 * v / 2, b1 / 2], [1 - b2, b1 * u, b1 * v, -b1],
              [-v, z, o, z], [(b2 - u / a) / 2, -(b1 * u - 1 / a) / 2, -b1 * v / 2, b1 / 2]]
        Rm = [[o, o, z, o], [u - a, u, z, u + a], [v, v, o, v], [H - u * a, q2 / 2, v, H + u * a]]

        def mul(M, x, there):
            x = x[[0, n, t, 3]] if there else x
            y = torch.stack([sum(M[i][j] * x[j] for j in range(4)) for i in range(4)])
            return y if there else y[[0, n, t, 3]]
        vl, dl, vr, dr, cl, cr = _both(c.geno_variant, [mul(Lm, q, 1) for q in Q], [mul(Lm, x, 1) for x in X], h)
        vl, dl, vr, dr = (mul(Rm, x, 0) for x in (vl, dl, vr, dr))
        chi = torch.minimum(torch.minimum(cl[0], cr[0]), torch.minimum(cl[3], cr[3]))
    vl, dl, chi = _safe(vl, dl, chi, Q[1])
    vr, dr, chi = _safe(vr, dr, chi, Q[2])
    return vl, dl, vr, dr, chi


class _Gas:
    """A Maxwellian with its normalised moments <u^a v^b xi^2c>; sign +-1: over u > 0 or u < 0."""

    def __init__(self, W, gamma):
        self.K = (4 - 2 * gamma) / (gamma - 1)
        self.r, self.U, self.V = W[0], W[1] / W[0], W[2] / W[0]
        self.p = (gamma - 1) * (W[3] - 0.5 * self.r * (self.U ** 2 + self.V ** 2))
        self.th = self.p / self.r
        self.u, self.v = self.table(torch.ones_like(self.U), self.U, self.U), self.table(torch.ones_like(self.U), self.V, self.V)
        self.xi = [1.0, self.K * self.th, self.K * (self.K + 2) * self.th ** 2]

    def table(self, t0, t1, m):
        t = [t0, t1]
        for n in range(5):
            t.append(m * t[-1] + (n + 1) * self.th * t[-2])
        return t

    def half(self, sign):
        x = self.U / torch.sqrt(2 * self.th)
        t0 = 0.5 * torch.special.erfc(-sign * x)
        return self.table(t0, self.U * t0 + sign * torch.sqrt(self.th / (2 * math.pi)) * torch.exp(-x * x), self.U)

    def psi(self, u, a, b, c=0):
        v, xi = self.v, self.xi
        m = lambda i, j, k: u[i] * v[j] * xi[k]  # noqa: E731
        return torch.stack([m(a, b, c), m(a + 1, b, c), m(a, b + 1, c),
                            0.5 * (m(a + 2, b, c) + m(a, b + 2, c) + m(a, b, c + 1))])

    def weighted(self, s, u, a, b):
        """<s u^a v^b psi>, s = s0 + s1 u + s2 v + s3 (u^2 + v^2 + xi^2) / 2"""
        return (s[0] * self.psi(u, a, b) + s[1] * self.psi(u, a + 1, b) + s[2] * self.psi(u, a, b + 1) +
                0.5 * s[3] * (self.psi(u, a + 2, b) + self.psi(u, a, b + 2) + self.psi(u, a, b, 1)))

    def slope(self, r):
        """s with <s psi> = r"""
        q = self.U ** 2 + self.V ** 2 + (self.K + 2) * self.th
        A, C, B = r[1] - self.U * r[0], r[2] - self.V * r[0], 2 * r[3] - q * r[0]
        s3 = (B - 2 * self.U * A - 2 * self.V * C) / (self.th ** 2 * (self.K + 2))
        s1, s2 = A / self.th - self.U * s3, C / self.th - self.V * s3
        return [r[0] - self.U * s1 - self.V * s2 - 0.5 * s3 * q, s1, s2, s3]


def _heat(F, W, U, V):
    return (F[3] - U * W[3] - U * F[1] - V * F[2] + (1.5 * U * U + 0.5 * V * V) * W[1] + U * V * W[2] -
            0.5 * U * (U * U + V * V) * W[0])


def _add_heat(c, F, W, U, V):
    return torch.cat([F[:3], (F[3] + (1 / c.Pr - 1) * _heat(F, W, U, V))[None]])


SWAP = [0, 2, 1, 3]


def _solve(c, dt, normal, Wl, Wr, Dl, Dr, Dt):
    """BGK interface solution: fitted F, F_t, one-sided W, W_t, each [4, ...] (Eq. eq:W-model)."""
    if normal:
        return [x[SWAP] for x in _solve(c, dt, 0, *(x[SWAP] for x in (Wl, Wr, Dl, Dr, Dt)))]
    l, r = _Gas(Wl, c.gamma), _Gas(Wr, c.gamma)
    ul, ur = l.half(1), r.half(-1)
    W0 = l.r * l.psi(ul, 0, 0) + r.r * r.psi(ur, 0, 0)
    g = _Gas(W0, c.gamma)
    al, bl, ar, br = l.slope(Dl / l.r), l.slope(Dt / l.r), r.slope(Dr / r.r), r.slope(Dt / r.r)
    a0, b0 = g.slope(0.5 * (Dl + Dr) / g.r), g.slope(Dt / g.r)
    tl, tr, t0 = (-(x.weighted(a, x.u, 1, 0) + x.weighted(b, x.u, 0, 1)) for x, a, b in ((l, al, bl), (r, ar, br), (g, a0, b0)))
    Al, Ar, A0 = l.slope(tl), r.slope(tr), g.slope(t0)
    tau = c.tau_c1 * dt + c.mu / g.p + c.tau_c2 * dt * (l.p - r.p).abs() / (l.p + r.p)
    cn, ct = [None] * 6, [None] * 6
    C = []
    for d in (0.5 * dt, dt):
        m = -torch.expm1(-d / tau)
        C.append((d - tau * m, -tau * d * (2 - m) + 2 * tau ** 2 * m, 0.5 * d * d - tau * d + tau ** 2 * m))
    for k, (n0, t1) in enumerate(((1.0, 0.0), (-tau, 0.0), (-tau, 1.0))):
        cn[k] = (4 * C[0][k] - C[1][k]) / dt
        ct[k] = 4 * (C[1][k] - 2 * C[0][k]) / dt ** 2
        cn[3 + k], ct[3 + k] = n0 - cn[k], t1 - ct[k]
    E = torch.exp(-dt / tau)
    e1 = -torch.expm1(-dt / tau)
    two = lambda f, h: l.r * f(l, ul, al, bl, Al) + r.r * f(r, ur, ar, br, Ar)  # noqa: E731
    flux = [g.r * g.psi(g.u, 1, 0), g.r * (g.weighted(a0, g.u, 2, 0) + g.weighted(b0, g.u, 1, 1)), g.r * g.weighted(A0, g.u, 1, 0),
            two(lambda s, u, a, b, A: s.psi(u, 1, 0), 0), two(lambda s, u, a, b, A: s.weighted(a, u, 2, 0) + s.weighted(b, u, 1, 1), 0),
            two(lambda s, u, a, b, A: s.weighted(A, u, 1, 0), 0)]
    cons = [W0, -g.r * t0, g.r * t0, W0,
            two(lambda s, u, a, b, A: s.weighted(a, u, 1, 0) + s.weighted(b, u, 0, 1), 0),
            two(lambda s, u, a, b, A: s.weighted(A, u, 0, 0), 0)]
    F, Ft, Wn, Wt = (sum(k * m for k, m in zip(q, v)) for q, v in ((cn, flux), (ct, flux), (cn, cons), (ct, cons)))
    F, Ft = _add_heat(c, F, Wn, g.U, g.V), _add_heat(c, Ft, Wt, g.U, g.V)
    return [F, Ft, e1 * Wn + E * Wl, e1 * Wn + E * Wr, e1 * Wt + E * l.r * tl, e1 * Wt + E * r.r * tr]


def _nodal(c, dt, W, Wx, Wy):
    g = _Gas(W, c.gamma)
    a, b = g.slope(Wx / g.r), g.slope(Wy / g.r)
    t = -(g.weighted(a, g.u, 1, 0) + g.weighted(b, g.u, 0, 1))
    A = g.slope(t)
    tau = c.tau_c1 * dt + c.mu / g.p
    out = []
    for i, j in ((1, 0), (0, 1)):
        Ft = g.r * g.weighted(A, g.u, i, j)
        F = g.r * g.psi(g.u, i, j) - tau * (g.r * (g.weighted(a, g.u, i + 1, j) + g.weighted(b, g.u, i, j + 1)) + Ft)
        if i:
            out += [_add_heat(c, F, W, g.U, g.V), _add_heat(c, Ft, g.r * t, g.U, g.V)]
        else:
            out += [_add_heat(c, F[SWAP], W[SWAP], g.V, g.U)[SWAP], _add_heat(c, Ft[SWAP], (g.r * t)[SWAP], g.V, g.U)[SWAP]]
    return out   # F, F_t, G, G_t


def _compact(c, chi, Fi, Fn):
    """Fluxes at the interfaces between consecutive entries along the last axis: Fi [.., n + 3], Fn [.., n + 2],
    chi [n + 1] -> the divergence's n differences."""
    low = Fi[..., 1:-1] if c.flux_variant == 62 else (8 * Fi[..., 1:-1] - Fn[..., :-1] - Fn[..., 1:]) / 6
    bar = (Fi[..., :-2] + 46 * Fi[..., 1:-1] + Fi[..., 2:] - 9 * (Fn[..., :-1] + Fn[..., 1:])) / 30
    f = (1 - chi) * low + chi * bar
    return f[..., 1:] - f[..., :-1]


def _ghost_rows(c, S, axis, dual, t, sides):
    """Three ghost layers at both ends of `axis` (0: x, the last one; 1: y) of S [12, ny, nx]."""
    S = S if axis == 0 else S.transpose(1, 2)
    n, other = S.shape[2], S.shape[1]
    ends = []
    for side in (0, 1):
        sd = 2 * axis + side
        ghost = [-3, -2, -1] if side == 0 else [n, n + 1, n + 2]

        def of(kind, W=None):
            if kind == 4:
                F = torch.zeros(12, other, 3, dtype=S.dtype, device=S.device)
                F[:4] = torch.tensor(W, dtype=S.dtype, device=S.device)[:, None, None]
                return F
            if kind == 0:
                src = [k % n for k in ghost]
            elif kind == 1:
                src = [0 if side == 0 else n - 1] * 3
            else:
                src = [(-k if dual else -k - 1) if side == 0 else ((2 * (n - 1) - k) if dual else 2 * n - 1 - k) for k in ghost]
            F = S[:, :, src]
            sg = torch.ones(12, dtype=S.dtype, device=S.device)
            if kind == 1:
                sg[4:] = 0
            elif kind >= 2:
                w = torch.ones(4, dtype=S.dtype, device=S.device)
                w[1 + axis] = -1
                if kind == 3:
                    w[2 - axis] = -1
                sg = torch.cat([w, -w if axis == 0 else w, -w if axis == 1 else w])
            return F * sg[:, None, None]
        if sides is None:
            ends.append(of(c.bc[sd]))
            continue
        s = sides[sd]
        W = []
        for q in s.get("prim", ((1.0, 0, 0, 1.0),) * 2):
            W.append([q[0], q[0] * q[1], q[0] * q[2], q[3] / (c.gamma - 1) + 0.5 * q[0] * (q[1] ** 2 + q[2] ** 2)])
        h, x0 = (c.hy, c.y0) if axis == 0 else (c.hx, c.x0)
        first = 0 if axis == 0 else -3
        pos = x0 + h * (torch.arange(other, dtype=S.dtype, device=S.device) + first + (0.0 if dual else 0.5))
        low = pos < s.get("split0", 0.0) + s.get("split_speed", 0.0) * t
        ends.append(torch.where(low[None, :, None], of(s["kind"][0], W[0]), of(s["kind"][1], W[1])))
    S = torch.cat([ends[0], S, ends[1]], dim=2)
    return S if axis == 0 else S.transpose(1, 2)


def _operator(c, dt, Sp, Sd, t):
    """Stage operator of both grids: L, L_t [4, ny, nx], gradients and their time derivatives [8, ny, nx]."""
    ny, nx, nyd, nxd = Sp.shape[1], Sp.shape[2], Sd.shape[1], Sd.shape[2]
    P, D = (_ghost_rows(c, _ghost_rows(c, S, 0, dual, t, c.sides), 1, dual, t, c.sides) for S, dual in ((Sp, 0), (Sd, 1)))
    h = (c.hx, c.hy)
    pts = []
    for typ in (0, 1):
        if typ == 0:
            R, C = nyd + 3, nx + 3
            l0 = [P[:, 1:1 + R, e:e + C] for e in range(4)]
            l1 = [D[:, e:e + R, 2:2 + C] for e in range(4)]
        else:
            R, C = ny + 3, nxd + 3
            l0 = [P[:, e:e + R, 1:1 + C] for e in range(4)]
            l1 = [D[:, 2:2 + R, e:e + C] for e in range(4)]
        rec = []
        for line, n in ((l0, typ), (l1, 1 - typ)):
            rec.append(_line(c, [x[:4] for x in line], [x[4 + 4 * n:8 + 4 * n] for x in line], h[n], n))
        tang = [0.5 * (r[1] + r[3]) for r in rec]
        o = [_solve(c, dt, n, r[0], r[2], r[1], r[3], tang[1 - k]) for k, (r, n) in enumerate(((rec[0], typ), (rec[1], 1 - typ)))]
        two = []
        for k in (0, 1):
            m, mt = (0.25 * (o[1 - k][q] + o[1 - k][q + 1]) for q in (2, 4))
            two.append(o[k][:2] + [0.5 * o[k][2] + m, 0.5 * o[k][3] + m, 0.5 * o[k][4] + mt, 0.5 * o[k][5] + mt, rec[k][4]])
        pts.append(two)
    (A0, A1), (B0, B1) = pts
    out = []
    for S, X, Y, n in ((P, [a[..., 2:2 + ny, :] for a in A0], [b[..., :, 2:2 + nx] for b in B0], (nx, ny)),
                       (D, [b[..., 1:1 + nyd, :] for b in B1], [a[..., :, 1:1 + nxd] for a in A1], (nxd, nyd))):
        W = S[:4, 2:-2, 2:-2]
        Wx = _node_derivative(c.geno_variant, [S[:4, 2:-2, e:e + n[0] + 2] for e in (1, 2, 3)], [S[4:8, 2:-2, e:e + n[0] + 2] for e in (1, 2, 3)], c.hx)
        Wy = _node_derivative(c.geno_variant, [S[:4, e:e + n[1] + 2, 2:-2] for e in (1, 2, 3)], [S[8:, e:e + n[1] + 2, 2:-2] for e in (1, 2, 3)], c.hy)
        F, Ft, G, Gt = _nodal(c, dt, W, Wx, Wy)
        Y = [y.transpose(-1, -2) for y in Y]
        G, Gt = G.transpose(1, 2), Gt.transpose(1, 2)
        L = [-_compact(c, X[6][..., 1:-1], X[q], f[:, 1:-1, :]) / c.hx - _compact(c, Y[6][..., 1:-1], Y[q], g[:, 1:-1, :]).transpose(1, 2) / c.hy
             for q, f, g in ((0, F, G), (1, Ft, Gt))]
        gr = [torch.cat([(X[q][..., 2:-1] - X[q + 1][..., 1:-2]) / c.hx, ((Y[q][..., 2:-1] - Y[q + 1][..., 1:-2]) / c.hy).transpose(1, 2)])
              for q in (2, 4)]
        out.append(L + gr)
    return out


def _walls(c, S):
    """Dual nodes on a no-slip wall: no velocity, no momentum gradients along the wall."""
    if 3 not in c.bc or c.sides is not None:
        return S
    ny, nx = S.shape[1:]
    m = torch.zeros(2, ny, nx, dtype=torch.bool, device=S.device)
    for side, (a, ix) in enumerate(((0, (slice(None), 0)), (0, (slice(None), -1)), (1, (0, slice(None))), (1, (-1, slice(None))))):
        if c.bc[side] == 3:
            m[a][ix] = True
    on = m[0] | m[1]
    z = torch.zeros_like(S[0])
    S = list(S.unbind(0))
    S[3] = torch.where(on, S[3] - 0.5 * (S[1] ** 2 + S[2] ** 2) / S[0], S[3])
    for f, w in ((1, on), (2, on), (9, m[0]), (10, m[0]), (5, m[1]), (6, m[1])):
        S[f] = torch.where(w, z, S[f])
    return torch.stack(S)


def _step(c, dt, S, t):
    """One S2O4 step of both grids (reading B of the gradient base)."""
    o1 = _operator(c, dt, *S, t)
    mid = []
    for (L, Lt, gb, gt), s, dual in zip(o1, S, (0, 1)):
        x = torch.cat([s[:4] + 0.5 * dt * L + 0.125 * dt * dt * Lt, gb + 0.5 * dt * gt])
        mid.append(_walls(c, x) if dual else x)
    o2 = _operator(c, dt, *mid, t + 0.5 * dt)
    new = []
    for (L, Lt, gb, _), (_, Lt2, _, gt2), s, dual in zip(o1, o2, S, (0, 1)):
        x = torch.cat([s[:4] + dt * L + dt * dt / 6 * (Lt + 2 * Lt2), gb + dt * gt2])
        new.append(_walls(c, x) if dual else x)
    return new


def _cfl(c, cfl, S):
    rate, nu = 0.0, 0.0
    for s in S:
        r, U, V = s[0], s[1] / s[0], s[2] / s[0]
        a = torch.sqrt(c.gamma * (c.gamma - 1) * (s[3] - 0.5 * r * (U * U + V * V)) / r)
        rate = max(rate, float(torch.maximum((U.abs() + a) / c.hx, (V.abs() + a) / c.hy).max()))
        nu = max(nu, float((c.mu / r).max()))
    dt = cfl / rate
    return min(dt, cfl * min(c.hx, c.hy) ** 2 / (8 * nu)) if nu > 0 else dt


def _pack(S):
    W, G, Wd, Gd = (torch.as_tensor(x).cuda() for x in S)
    return [torch.cat([W, G.reshape(8, *G.shape[2:])]), torch.cat([Wd, Gd.reshape(8, *Gd.shape[2:])])]


def _unpack(S):
    return [x for s in S for x in (s[:4], s[4:].reshape(2, 4, *s.shape[1:]))]


def _advance(c, S, steps, cfl=None, dt=None):
    t = 0.0
    for _ in range(steps):
        d = dt if cfl is None else _cfl(c, cfl, S)
        S = _step(c, d, S, t)
        t += d
    return S, t


def _line_operator(c, dt, S):
    """Stage operator of lines S [6, batch, n] (rho, rho U, rho E and their averaged gradients)."""
    n = S.shape[2]
    full = torch.zeros(12, S.shape[1], n, dtype=S.dtype, device=S.device)
    full[[0, 1, 3, 4, 5, 7]] = S
    P = _ghost_rows(c, full, 0, 0, 0.0, None)
    e = [P[:, :, k:k + n + 3] for k in range(4)]
    vl, dl, vr, dr, chi = _line(c, [x[:4] for x in e], [x[4:8] for x in e], c.hx, 0)
    o = _solve(c, dt, 0, vl, vr, dl, dr, torch.zeros_like(vl))
    Wx = _node_derivative(c.geno_variant, [P[:4, :, k:k + n + 2] for k in (1, 2, 3)], [P[4:8, :, k:k + n + 2] for k in (1, 2, 3)], c.hx)
    F, Ft, _, _ = _nodal(c, dt, P[:4, :, 2:-2], Wx, torch.zeros_like(Wx))
    L, Lt = (-_compact(c, chi[:, 1:-1], o[q], f) / c.hx for q, f in ((0, F), (1, Ft)))
    gb, gt = ((o[q][..., 2:-1] - o[q + 1][..., 1:-2]) / c.hx for q in (2, 4))
    return [x[[0, 1, 3]] for x in (L, Lt, gb, gt)]


def _line_step(c, dt, S):
    L, Lt, gb, gt = _line_operator(c, dt, S)
    _, Lt2, _, gt2 = _line_operator(c, dt, torch.cat([S[:3] + 0.5 * dt * L + 0.125 * dt * dt * Lt, gb + 0.5 * dt * gt]))
    return torch.cat([S[:3] + dt * L + dt * dt / 6 * (Lt + 2 * Lt2), gb + dt * gt2])


def exact(case, seed):
    kind = case["kind"]
    if kind == "lines":
        c, W, X, cfl, dt = _line_problem(case, seed)
        S = torch.cat([torch.from_numpy(a).cuda().transpose(0, 1) for a in (W, X)])
        t, k = 0.0, 0
        while k < case["steps"] if case["loop"] == "fixed" else t < case["t_end"] * (1 - 1e-14):
            if case["loop"] != "fixed":
                U = S[1] / S[0]
                a = torch.sqrt(c.gamma * (c.gamma - 1) * (S[2] / S[0] - 0.5 * U * U))
                dt = min(cfl / float(((U.abs() + a) / c.hx).max()), case["t_end"] - t)
            S = _line_step(c, dt, S)
            t += dt
            k += 1
        S = _snapshot(case, [S[:3].transpose(0, 1).contiguous(), S[3:].transpose(0, 1).contiguous()], c.hx, torch.float64)
        return S + [np.array([k], dtype=np.int32)] if case["loop"] == "run" else S
    if kind == "ensemble":
        if case["members"] * case["steps"] > 200:   # over 20 s
            return None
        flat, times = [], []
        for c in _members(case, seed):
            S, t = _advance(c, _pack(c.initial_state()), case["steps"], cfl=0.2)
            flat += [x.reshape(-1) for x in _snapshot(case, _unpack(S), (c.hx, c.hy), torch.float64)]
            times.append(t)
        return [torch.cat(flat), np.array(times), np.zeros(len(times), dtype=np.int32)]
    c, cfl, dt = _problem(case, seed)
    S = _pack(c.initial_state())
    if kind == "adjoint":
        lam = torch.zeros_like(S[0])
        lam[0] = torch.from_numpy(_misfit(c, seed)).cuda()
        lam = [lam, torch.zeros_like(S[1])]
        states = [S]
        with torch.no_grad():
            for _ in range(case["steps"] - 1):
                states.append(_step(c, dt, states[-1], 0.0))
        for S in reversed(states):
            S = [x.detach().requires_grad_(True) for x in S]
            lam = torch.autograd.grad(_step(c, dt, S, 0.0), S, lam)
        return _unpack(lam)
    S, _ = _advance(c, S, case["steps"], **(dict(cfl=cfl) if case["loop"] == "cfl" else dict(dt=dt)))
    out = _snapshot(case, _unpack(S), (c.hx, c.hy), torch.float64)
    return [x.cpu() for x in out] if case["io"] == "host" else out
