"""Steps, the stage operator and get_state can be captured into a CUDA graph in
both precisions, programmatic launches included; the replay gives the bits of
the calls themselves."""
import pytest

from paper_2606_17772_gb300 import fdcgks, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

CASES = [inputs.vortex(17), inputs.vortex(330), inputs.random_smooth(61, 14, seed=9, amp=0.05, bc=(3, 3, 3, 2), mu=0.01)]


@pytest.mark.parametrize("precision", [fdcgks.FP64, fdcgks.MIXED])
@pytest.mark.parametrize("k", range(len(CASES)))
def test_captured_steps_equal_the_calls(k, precision):
    S = [torch.from_numpy(a).cuda() for a in CASES[k].initial_state()]
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        with fdcgks.Solver.from_case(CASES[k], precision) as s:
            s.set_state(*S)
            dt = s.cfl_dt(0.1)
            s.steps(dt, 4)
            ref = s.get_state()
            s.set_state(*S)
            out = [torch.empty_like(a) for a in ref]
            st.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                s.steps(dt, 2)
                s.get_state(out)
            for _ in range(2):
                graph.replay()
            st.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(ref, out))
            assert not s.check()
