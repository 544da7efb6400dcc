"""The mixed update's forms (1, 2 or 4 rows a thread by the grid's size) give the
same bits: rough data that repeat along the periodic directions stay a repetition
of the small grid's step on grids of the other size classes, whose edges of rows
and of tiles lie elsewhere in the pattern.  Class timing is on, so that every
size runs the same nodal and point kernels."""
import numpy as np
import pytest

from paper_2606_17772_gb300 import fdcgks, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

H = 1.0 / 32   # spacings and quotients exact


def advance(nx, ny, bc, state, grad_base, steps=3):
    case = inputs.Case("tiled", nx, ny, 0.0, nx * H, 0.0, ny * H, bc, mu=0.01, tau_c2=1.0, grad_base=grad_base)
    with fdcgks.Solver.from_case(case, fdcgks.MIXED) as s:
        s.set_state(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in state])
        s.set_profiling(True)
        s.steps(2.0 ** -10, steps)
        assert not s.check()
        return [t.cpu().numpy() for t in s.get_state()]


def rough(nx, ny, bc, seed):
    rng = np.random.default_rng(seed)
    out = []
    for dual in (0, 1):
        w, h = nx + (dual and bc[0] != 0), ny + (dual and bc[2] != 0)
        rho, U, V, p = (c + 0.2 * rng.uniform(-1, 1, size=(h, w)) for c in (1.0, 0.3, -0.2, 1.0))
        out.append(np.stack([rho, rho * U, rho * V, p / 0.4 + 0.5 * rho * (U * U + V * V)]))
        out.append(2.0 * rng.normal(size=(2, 4, h, w)))
    return out


# base grid, boundary kinds, repetitions along x and y: 1 row below 29,000 nodes, 2 up to 100,000, 4 above;
# the last rows hold 1, 2 or 3 of a thread's rows
TILED = [(31, 31, (0, 0, 0, 0), [(6, 7), (7, 6), (11, 11), (10, 12), (9, 13), (8, 14)]),
         (93, 31, (3, 2, 0, 0), [(1, 11), (1, 35), (1, 36)]),       # a dual row is wider by one
         (31, 93, (0, 0, 2, 3), [(12, 1), (36, 1)]),                # 93 primary rows, 94 dual rows
         (31, 94, (0, 0, 3, 3), [(12, 1), (36, 1)])]


@pytest.mark.parametrize("grad_base", [0, 1])
@pytest.mark.parametrize("nx,ny,bc,reps", TILED)
def test_forms_agree_to_the_bit(nx, ny, bc, reps, grad_base):
    base = rough(nx, ny, bc, seed=nx + ny)
    ref = advance(nx, ny, bc, base, grad_base)
    for kx, ky in reps:
        def tile(a):
            return np.tile(a, (1,) * (a.ndim - 2) + (ky, kx))
        out = advance(kx * nx, ky * ny, bc, [tile(a) for a in base], grad_base)
        for a, b in zip(out, ref):
            np.testing.assert_array_equal(a, tile(b))
