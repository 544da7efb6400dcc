"""The FP64 reconstructions keep their range: lines with differences up to 1e37
(GENO's text constants, whose path function takes the eighth power of them)
give what the same lines scaled down by a power of two give."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "librange.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_2606_17772_gb300", "csrc"), "-I", HERE, "-o", out,
                    os.path.join(HERE, "geno_screen_probe.cpp")], check=True)
    return ctypes.CDLL(out)


def _run(probe, variant, rows):
    out, ref = np.zeros((len(rows), 7)), np.zeros((len(rows), 7))
    D = ctypes.POINTER(ctypes.c_double)
    probe.probe_screen(variant, ctypes.c_double(0.5), len(rows), rows.ctypes.data_as(D), out.ctypes.data_as(D),
                       ref.ctypes.data_as(D))
    return out


# largest exponents: (sum of three weights) 10 (5.4 d^2)^4 and the path function's (5.4 d^2)^2r stay below 2^1024
@pytest.mark.parametrize("variant,exponents", [(0, (100, 112, 114, 120, 122)), (1, (70, 80))])
def test_large_differences_scale(probe, variant, exponents):
    rng = np.random.default_rng(variant)
    rows = rng.uniform(-1, 1, size=(500, 8))
    rows[::5, :4] = [0.0, 0.0, 1.0, 1.0] + 1e-3 * rows[::5, 4:]      # a jump
    rows[::5, 4:] *= 1e-2
    base = _run(probe, variant, rows * 2.0 ** 55)     # eps_a and eps_w are below an ulp of the indicators here
    assert np.isfinite(base).all() and (base[:, 2] < 1).any()
    values = [0, 1, 3, 4, 6]
    for e in exponents:
        out = _run(probe, variant, rows * 2.0 ** e)
        np.testing.assert_array_equal(out[:, values], base[:, values] * 2.0 ** (e - 55))
        np.testing.assert_array_equal(out[:, [2, 5]], base[:, [2, 5]])
