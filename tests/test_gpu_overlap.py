"""Mixed steps launch their kernels as programmatic dependents: steps queued
back to back give, bit for bit, what steps with a synchronisation after each
give, also with the CFL reduction between them and on two streams at once."""
import pytest

from paper_2606_17772_gb300 import fdcgks, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

CASES = [inputs.vortex(17), inputs.vortex(130), inputs.vortex(330),
         inputs.random_smooth(61, 14, seed=9, amp=0.05, bc=(3, 3, 3, 2), mu=0.01)]


def run(case, precision, apart, stream=None):
    with torch.cuda.stream(stream or torch.cuda.current_stream()):
        s = fdcgks.Solver.from_case(case, precision)
        s.set_state(*[torch.from_numpy(a).cuda() for a in case.initial_state()])
        for _ in range(3):
            dt = s.cfl_dt(0.2)
            if apart:
                for _ in range(4):
                    s.step(dt)
                    torch.cuda.synchronize()
            else:
                s.steps(dt, 4)
        assert not s.check()
        return s, s.get_state()


@pytest.mark.parametrize("precision", [fdcgks.FP64, fdcgks.MIXED])
@pytest.mark.parametrize("k", range(len(CASES)))
def test_queued_steps_equal_synchronised_ones(k, precision):
    a, b = run(CASES[k], precision, True)[1], run(CASES[k], precision, False)[1]
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(a, b))


def test_two_streams():
    ref = [run(c, fdcgks.MIXED, True)[1] for c in CASES[:2]]
    out = [run(c, fdcgks.MIXED, False, torch.cuda.Stream())[1] for c in CASES[:2]]
    torch.cuda.synchronize()
    for r, o in zip(ref, out):
        assert all(torch.equal(x, y) for x, y in zip(r, o))
