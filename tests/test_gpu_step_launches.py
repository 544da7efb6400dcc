"""Programmatic dependent launches inside a mixed step: the same kernels with
ordinary launches (a switch of one context, for tests) give the same bits, alone
and with two streams busy at once."""
import ctypes

import pytest

from paper_2606_17772_gb300 import fdcgks, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

# merged and separate nodes and points, every update form, both CFL reductions, split sides, walls
CASES = [inputs.vortex(9), inputs.vortex(33), inputs.vortex(130), inputs.vortex(180), inputs.vortex(330),
         inputs.random_smooth(61, 14, seed=9, amp=0.05, bc=(3, 3, 3, 2), mu=0.01),
         inputs.random_smooth(300, 400, seed=5, amp=0.05, bc=(1, 1, 3, 3), mu=0.01), inputs.double_mach(96, 24)]


def solver(case, overlap):
    s = fdcgks.Solver.from_case(case, fdcgks.MIXED)
    assert fdcgks.load().fdk_set_overlap(s._h, ctypes.c_int(overlap)) == 0
    s.set_state(*[torch.from_numpy(a).cuda() for a in case.initial_state()])
    return s


def queue(s, dt, rounds):
    """CFL reductions between the steps, whose result nothing waits for but the call itself."""
    out = []
    for _ in range(rounds):
        s.steps(dt, 3)
        out.append(s.cfl_dt(0.2))
    s.steps(dt, 2)
    return out


def step_size(case):
    with solver(case, 0) as s:
        return s.cfl_dt(0.1)


@pytest.mark.parametrize("k", range(len(CASES)))
def test_overlapped_launches_equal_ordinary_ones(k):
    dt = step_size(CASES[k])
    with solver(CASES[k], 0) as s:
        cfl = queue(s, dt, 3)
        ref = s.get_state()
        assert not s.check()
    for _ in range(4):
        with solver(CASES[k], 1) as s:
            assert queue(s, dt, 3) == cfl
            out = s.get_state()
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(ref, out))


@pytest.mark.parametrize("pair", [(1, 4), (2, 6), (3, 3), (5, 7)])
def test_two_busy_streams(pair):
    cases = [CASES[k] for k in pair]
    n, ref = 12, []
    for c in cases:
        with solver(c, 0) as s:
            s.steps(step_size(c), n)
            ref.append(s.get_state())
            torch.cuda.synchronize()
    dts = [step_size(c) for c in cases]
    streams = [torch.cuda.Stream() for _ in cases]
    runs = []
    for c, st in zip(cases, streams):
        with torch.cuda.stream(st):
            runs.append(solver(c, 1))
    torch.cuda.synchronize()
    hold = torch.cuda.Event()
    filler = torch.empty(1 << 28, dtype=torch.float32, device="cuda")
    for _ in range(4):
        filler.fill_(1.0)          # the streams' work queues up behind this
    hold.record()
    for st in streams:
        st.wait_event(hold)
    for part in range(n // 3):     # both queues are filled before either run is waited for
        for s, dt in zip(runs, dts):
            s.steps(dt, 3)
    out = []
    for s, st in zip(runs, streams):
        with torch.cuda.stream(st):
            out.append(s.get_state())
    torch.cuda.synchronize()
    for r, o in zip(ref, out):
        assert all(torch.equal(a, b) for a, b in zip(r, o))
    assert not any(s.check() for s in runs)
