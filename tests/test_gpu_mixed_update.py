"""The mixed update's forms (1, 2 or 4 rows a thread by the grid's size; 4 in
an ensemble, whose tiles may be any width) give the same step: a single run
against an ensemble member, at the edges of rows, warps and size classes, with
walls (components coupled) and both gradient bases."""
import numpy as np
import pytest

from paper_2606_17772_gb300 import fdcgks, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

SIZES = [(1, 1, (0, 0, 0, 0)), (31, 3, (3, 3, 3, 3)), (32, 5, (2, 3, 0, 0)), (33, 6, (0, 0, 3, 2)), (65, 7, (1, 1, 3, 3)),
         (170, 170, (0, 0, 0, 0)), (171, 170, (3, 2, 3, 2)), (319, 318, (3, 3, 3, 3))]


@pytest.mark.parametrize("lbx", [0, 3, 5, 7])
@pytest.mark.parametrize("grad_base", [0, 1])
@pytest.mark.parametrize("nx,ny,bc", SIZES)
def test_single_run_equals_member(nx, ny, bc, grad_base, lbx):
    case = inputs.random_smooth(nx, ny, seed=nx + ny, amp=0.05, bc=bc, mu=0.01, grad_base=grad_base)
    S0 = [torch.from_numpy(a).cuda() for a in case.initial_state()]
    with fdcgks.Solver.from_case(case, fdcgks.MIXED) as s:
        s.set_state(*S0)
        dt = s.cfl_dt(0.3)
        s.steps(dt, 2)
        assert not s.check()
        ref = [t.cpu().numpy() for t in s.get_state()]
    with fdcgks.Ensemble.from_cases([case], fdcgks.MIXED) as e:
        e.set_tiles([5, 5, lbx, 0])
        e.set_state(0, *S0)
        e.run(2, dt=[dt])
        out = [np.asarray(t) for t in e.get_state(0, device=False)]
    # the same per-node arithmetic in several kernels: equal up to the fusing of
    # multiply-adds, a few ulp of the state a step, over h for gradients
    u, h = 2.0 ** -24, min(case.hx, case.hy)
    for k, (a, b) in enumerate(zip(out, ref)):
        scale = max(np.abs(ref[k - k % 2]).max(), 1.0)
        assert np.isfinite(a).all()
        assert np.abs(a - b).max() <= 1e3 * u * scale * (1.0 if k % 2 == 0 else 1.0 / h)
