"""Ghosts of a line are written by the threads that update the nodes they copy
(and once when a call starts): the shortest lines, where one node feeds several
ghosts, and every pair of ends, against the oracle and against one call a step."""
import numpy as np
import pytest

import oracle
from paper_2606_17772_gb300 import fdcgks, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

ENDS = [(n, (0, 0)) for n in (1, 2, 3, 4, 7, 32, 33)] + [(n, e) for n in (3, 4, 5, 31, 64) for e in
                                                         ((1, 1), (2, 2), (1, 2), (2, 1))]


@pytest.mark.parametrize("n,ends", ENDS)
def test_short_lines_and_every_end(n, ends):
    case = inputs.random_smooth(n, 1, seed=n, amp=0.1, bc=ends + (0, 0), tau_c1=0.05, tau_c2=1.0)
    W, G = inputs.line_state(case)
    ref = oracle.steps_1d(oracle.make_params(**case.oracle_kwargs()), 0.002, 3, W, G)
    out = []
    for calls in (1, 3):
        with fdcgks.Lines.from_case(case) as L:
            L.set_state(W, G)
            for _ in range(calls):
                L.steps(0.002, 3 // calls)
            assert L.check()[0][0] == 0
            out.append(L.get_state(device=False))
    for a, b, r in zip(out[0], out[1], ref):
        assert np.array_equal(a, b)
        # the steps' tolerance of test_gpu_line.py: 1e-12 a step, relative to the group
        s = np.abs(r).max()
        assert np.abs(a[0] - r).max() <= 3e-12 * (s if s > 0 else 1.0)
