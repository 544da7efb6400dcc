"""State arrays that no kernel reads directly (here pinned host memory handed
over as device arrays, which takes the way of a second GPU's memory) load, read
back and differentiate like ordinary device arrays, bit for bit; and a get_state
into device arrays can still be captured."""
import ctypes

import pytest

from paper_2606_17772_gb300 import fdcgks, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

PRECISIONS = [fdcgks.FP64, fdcgks.MIXED]


def ptrs(arrs):
    return [ctypes.c_void_p(a.data_ptr()) for a in arrs]


def state(case):
    S = [torch.from_numpy(a).contiguous() for a in case.initial_state()]
    return [a.cuda() for a in S], [a.pin_memory() for a in S]


def same(a, b):
    torch.cuda.synchronize()
    return all(torch.equal(x.cpu(), y.cpu()) for x, y in zip(a, b))


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("nx,ny", [(3, 4), (33, 17)])
def test_solver(nx, ny, precision):
    case = inputs.random_smooth(nx, ny, seed=nx, amp=0.05, bc=(3, 2, 0, 0), mu=0.01)
    dev, pin = state(case)
    lib = fdcgks.load()
    with fdcgks.Solver.from_case(case, precision) as s:
        s.set_state(*dev)
        s.steps(1e-3, 2)
        ref = s.get_state()
        assert lib.fdcgks_set_state(s._h, *ptrs(pin), 1) == 0
        s.steps(1e-3, 2)
        out = [torch.empty_like(a).pin_memory() for a in pin]
        assert lib.fdcgks_get_state(s._h, *ptrs(out), 1) == 0
        assert same(ref, out)


@pytest.mark.parametrize("precision", PRECISIONS)
def test_ensemble(precision):
    cases = [inputs.vortex(8), inputs.random_smooth(13, 29, seed=3, amp=0.05, bc=(0, 0, 3, 3), mu=0.01)]
    lib = fdcgks.load()
    with fdcgks.Ensemble.from_cases(cases, precision) as e:
        for m, c in enumerate(cases):
            dev, pin = state(c)
            assert lib.fdcgks_ens_set_state(e._h, m, *ptrs(pin), 1) == 0
            out = [torch.empty_like(a).pin_memory() for a in pin]
            assert lib.fdcgks_ens_get_state(e._h, m, *ptrs(out), 1) == 0
            e.set_state(m, *dev)
            assert same(e.get_state(m, device=True), out)


@pytest.mark.parametrize("precision", PRECISIONS)
def test_adjoint(precision):
    case = inputs.random_smooth(15, 13, seed=40, amp=0.08, tau_c1=0.05, tau_c2=1.0)
    dev, pin = state(case)
    g = torch.Generator().manual_seed(1)
    seed = [torch.randn(a.shape, dtype=torch.float64, generator=g).pin_memory() for a in pin]
    out = [torch.empty_like(a).pin_memory() for a in pin]
    lib = fdcgks.load()
    with fdcgks.Solver.from_case(case, precision) as s:
        ref = s.vjp_steps(0.01, 3, dev, [a.cuda() for a in seed], checkpoint_every=2)
        assert lib.fdcgks_vjp_steps(s._h, ctypes.c_double(0.01), 3, 2, *ptrs(pin), *ptrs(seed), *ptrs(out)) == 0
    torch.cuda.synchronize()
    for a, b in zip(ref, out):   # the order of the atomic additions differs between runs
        assert (a.cpu() - b).abs().max() <= 1e-12 * a.abs().max().cpu()


@pytest.mark.parametrize("precision", PRECISIONS)
def test_lines(precision):
    case = inputs.lax_strip(30, 1)
    W, Wx = (torch.from_numpy(a).contiguous() for a in inputs.line_state(case))
    lib = fdcgks.load()
    with fdcgks.Lines.from_case(case, precision=precision) as L:
        L.set_state(W.cuda()[None], Wx.cuda()[None])
        L.steps(1e-3, 2)
        ref = L.get_state()
        pin = [W.pin_memory(), Wx.pin_memory()]
        assert lib.fdcgks_line_set_state(L._h, *ptrs(pin), 1) == 0
        L.steps(1e-3, 2)
        out = [torch.empty_like(a, device="cpu").pin_memory() for a in ref]
        assert lib.fdcgks_line_get_state(L._h, *ptrs(out), 1) == 0
        assert same(ref, out)


def test_get_state_is_captured():
    case = inputs.vortex(16)
    dev, _ = state(case)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = fdcgks.Solver.from_case(case)
        s.set_state(*dev)
        out = [torch.zeros_like(a) for a in dev]
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            s.get_state(out)
        graph.replay()
    torch.cuda.synchronize()
    assert same(out, dev)
