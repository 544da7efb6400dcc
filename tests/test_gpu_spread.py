"""Results that rounding moves, with bounds taken from the oracle's own spread
instead of from one build: the transpose test of viscous walls, the Sod line's
minimum and the blast waves' density peak."""
import numpy as np
import pytest

import oracle
from paper_2606_17772_gb300 import fdcgks, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def dot(a, b):
    return float(sum(np.vdot(x, y) for x, y in zip(a, b)))


@pytest.mark.parametrize("nsteps", [1, 3])
def test_walls_viscous_linear_transpose(nsteps):
    """The adjoint against the oracle's central differences at steps of 1e-7 to
    1e-6, where they agree among themselves to 1e-7 of their value (at 1e-8
    rounding moves them by 4e-6, at 1e-5 truncation by 2e-4)."""
    case, dt = inputs.random_smooth(13, 11, seed=41, amp=0.06, bc=(3, 3, 3, 2), mu=0.01, Pr=0.73, tau_c2=1.0,
                                    geno_variant=2), 0.004
    S0 = case.initial_state()
    rng = np.random.default_rng(7)
    v = [rng.standard_normal(a.shape) * (np.abs(a).max() + 1e-3) for a in S0]
    seed = [rng.standard_normal(a.shape) for a in S0]
    p = oracle.make_params(**case.oracle_kwargs())
    fd = []
    for eps in (1e-7, 3e-7, 1e-6):
        up, down = (oracle.steps(p, dt, nsteps, *[a + e * b for a, b in zip(S0, v)]) for e in (eps, -eps))
        fd.append(dot(seed, [(x - y) / (2 * eps) for x, y in zip(up, down)]))
    spread = max(fd) - min(fd)
    assert spread <= 2e-7 * abs(fd[1])
    with fdcgks.Solver.from_case(case) as s:
        g = s.vjp_steps(dt, nsteps, *[[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in x] for x in (S0, seed)],
                        checkpoint_every=2)
        ad = dot([t.cpu().numpy() for t in g], v)
    assert abs(ad - fd[1]) <= 3 * spread, (ad, fd)


# the oracle over 13 runs (the initial values, and 12 times 1 + 1e-15 N(0, 1) of them): the least density of the
# Sod line over 0.125 was 0.9871 to 0.9987, the blast waves' density peak 5.539 to 5.877; a run may lie a width outside
SOD_MIN = (0.9871, 0.9987)
BLAST_PEAK = (5.539, 5.877)


def widened(lo, hi):
    return lo - (hi - lo), hi + (hi - lo)


def line(case, precision, t, cfl):
    W, G = inputs.line_state(case)
    with fdcgks.Lines.from_case(case, precision=precision) as L:
        L.set_state(W, G)
        L.run(t, cfl)
        assert L.check()[1] == 0
        return L.get_state(device=False)[0][0][0]


@pytest.mark.parametrize("precision", [fdcgks.FP64, fdcgks.MIXED])
def test_sod_line_minimum(precision):
    rho = line(inputs.sod_strip(200, 1), precision, 0.2, 0.3)
    lo, hi = widened(*SOD_MIN)
    assert lo <= rho.min() / 0.125 <= hi


@pytest.mark.parametrize("precision", [fdcgks.FP64, fdcgks.MIXED])
def test_blast_wave_peak(precision):
    rho = line(inputs.woodward_colella(400, flux_variant=62, geno_variant=1), precision, 0.038, 0.4)
    lo, hi = widened(*BLAST_PEAK)
    assert lo <= rho.max() <= hi
