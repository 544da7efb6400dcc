"""The stage's launch forms give the same step: nodes and interface points in
one launch (small grids; FP64 always) or apart (class timing switched on).
Sizes at the edges of warps and tiles, every grid kind, both precisions and
both reconstructions."""
import numpy as np
import pytest

from paper_2606_17772_gb300 import fdcgks, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

SIZES = [(1, 1, (0, 0, 0, 0)), (3, 3, (2, 2, 3, 3)), (13, 1, (1, 2, 0, 0)), (14, 30, (0, 0, 2, 2)), (29, 13, (1, 1, 3, 2)),
         (30, 29, (0, 0, 0, 0)), (61, 14, (3, 3, 3, 2))]


@pytest.mark.parametrize("char", [0, 1])
@pytest.mark.parametrize("prec", [fdcgks.FP64, fdcgks.MIXED])
@pytest.mark.parametrize("nx,ny,bc", SIZES)
def test_merged_and_separate_launches_agree(nx, ny, bc, prec, char):
    case = inputs.random_smooth(nx, ny, seed=nx + ny, amp=0.05, bc=bc, tau_c1=0.05, tau_c2=1.0, recon_vars=char)
    S0 = [torch.from_numpy(a).cuda() for a in case.initial_state()]
    out = []
    for apart in (False, True):
        with fdcgks.Solver.from_case(case, prec) as s:
            s.set_profiling(apart)
            s.set_state(*S0)
            s.steps(0.002, 2)
            assert not s.check()
            out.append([t.cpu().numpy() for t in s.get_state()])
    # the same per-node arithmetic compiled into two kernels: equal up to the
    # fusing of multiply-adds, a few ulp of the state a step, over h for gradients
    u = 2.0 ** -53 if prec == fdcgks.FP64 else 2.0 ** -24
    h = min(case.hx, case.hy)
    for k, (a, b) in enumerate(zip(*out)):
        scale = max(np.abs(out[1][k - k % 2]).max(), 1.0)
        assert np.isfinite(a).all()
        assert np.abs(a - b).max() <= 1e3 * u * scale * (1.0 if k % 2 == 0 else 1.0 / h)
