"""The FP64 path decides GENO's saturation by an FP32 estimate with margins
first; that must never skip an indicator that FP64 would have used.  The
reconstructions with the screen are compared with the same arithmetic without
it (the dual numbers' instantiation) on lines that cross the decision's
threshold at every scale, down to underflow and up to overflow of FP32."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(ROOT, "paper_2606_17772_gb300", "csrc")


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "libscreen.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-I", CSRC, "-I", HERE, "-o",
                    out, os.path.join(HERE, "geno_screen_probe.cpp")], check=True)
    return ctypes.CDLL(out)


def _lines(rng, scale, curve):
    """Q, Q_x h of a line with gradient ~ scale and curvature ~ curve * scale (curve ~ 0.1 is the threshold)."""
    a, b, c = rng.normal(size=3) * scale
    x = np.arange(4.0)
    Q = a * x + 0.5 * curve * b * x * x + 0.1 * curve * c * x ** 3
    G = a + curve * b * x + 0.3 * curve * c * x * x
    return np.concatenate([Q, G * (1 + 0.3 * curve * rng.normal(size=4))])


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("scale", [1e-30, 1e-16, 1e-8, 1e-6, 1e-3, 1.0, 1e6, 1e19, 1e40])
def test_screen_skips_only_saturated_indicators(probe, variant, scale):
    rng = np.random.default_rng([variant, int(np.log10(scale) + 50)])
    h, n = 0.05, 4000
    rows = np.array([_lines(rng, scale, 10.0 ** rng.uniform(-3, 1)) for _ in range(n)])
    rows[:, 4:] /= h
    rows[:8] = 0.0
    a, b = np.zeros((n, 7)), np.zeros((n, 7))
    D = ctypes.POINTER(ctypes.c_double)
    probe.probe_screen(variant, ctypes.c_double(h), n, rows.ctypes.data_as(D), a.ctypes.data_as(D), b.ctypes.data_as(D))
    # without contraction the two builds round alike, so what the screen decides is the only difference;
    # at 1e40 the cubes of the indicators stay below FP64's overflow
    ok = np.isfinite(b).all(axis=1)
    assert ok.sum() > n // 2
    np.testing.assert_array_equal(a[ok], b[ok])
    chi = b[ok][:, [2, 5]]
    if 1e-6 < scale < 1e19:
        assert (chi == 1.0).any() and (chi < 1.0).any()   # both sides of the threshold were met
