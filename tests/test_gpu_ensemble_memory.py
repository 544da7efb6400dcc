"""An ensemble holds its members' buffers and no second copy of a state: host
arrays are staged in the members' own point buffers, and pass through them
unchanged before and after steps."""
import numpy as np
import pytest

from paper_2606_17772_gb300 import fdcgks, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("precision", [fdcgks.FP64, fdcgks.MIXED])
def test_memory_of_the_members_only(precision):
    case = inputs.vortex(1024)
    pitch, rows = (1024 + 6 + 31) // 32 * 32, 1024 + 6
    ppitch, prows = (1024 + 3 + 31) // 32 * 32, 1024 + 3
    # per padded node: states, accumulators, gradient bases and nodal fluxes of both grids; 2 x 50 values a point
    values, size = (2 * (12 + 12 + 4 + 8 + 16), 8) if precision == fdcgks.FP64 else (2 * (36 + 8 + 16 + 16), 4)
    members = size * (values * pitch * rows + 100 * ppitch * prows)
    torch.cuda.synchronize()
    used = members * 2
    for _ in range(5):     # the least of a few: other processes on the device allocate too
        free = torch.cuda.mem_get_info()[0]
        with fdcgks.Ensemble.from_cases([case], precision):
            used = min(used, free - torch.cuda.mem_get_info()[0])
    assert used <= members + 32 * 2 ** 20     # a padded FP64 state of both grids would be 208 MB more


@pytest.mark.parametrize("precision", [fdcgks.FP64, fdcgks.MIXED])
def test_host_arrays_pass_unchanged(precision):
    cases = [inputs.vortex(9), inputs.random_smooth(40, 23, seed=2, amp=0.05, bc=(3, 2, 1, 1), mu=0.01), inputs.vortex(64)]
    with fdcgks.Ensemble.from_cases(cases, precision) as e:
        for m, c in enumerate(cases):
            e.set_state(m, *c.initial_state())
        for steps in (0, 3):
            if steps:
                e.run(steps, cfl=0.2)
            for m in range(len(cases)):
                host, dev = e.get_state(m, device=False), e.get_state(m, device=True)
                for a, b in zip(host, dev):
                    assert np.array_equal(np.asarray(a), b.cpu().numpy())
                e.set_state(m, *host)
                for a, b in zip(host, e.get_state(m, device=False)):
                    assert np.array_equal(np.asarray(a), np.asarray(b))
