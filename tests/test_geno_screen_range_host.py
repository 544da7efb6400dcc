"""The FP32 saturation screen at any spacing: where FP32 cannot hold the spacing
or flushes gradients that still count, it must leave the decision to FP64."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))
D = ctypes.POINTER(ctypes.c_double)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "libscreenrange.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_2606_17772_gb300", "csrc"), "-I", HERE, "-o", out,
                    os.path.join(HERE, "geno_screen_probe.cpp")], check=True)
    return ctypes.CDLL(out)


def _lines(rng, scale, curve):
    """Q, Q_x h of a line with gradient ~ scale and curvature ~ curve * scale (curve ~ 0.1 is the threshold)."""
    a, b, c = rng.normal(size=3) * scale
    x = np.arange(4.0)
    Q = a * x + 0.5 * curve * b * x * x + 0.1 * curve * c * x ** 3
    G = a + curve * b * x + 0.3 * curve * c * x * x
    return np.concatenate([Q, G * (1 + 0.3 * curve * rng.normal(size=4))])


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("h", [1e-300, 1e-44, 3e-42, 1e-38, 1e-30, 1.0, 1e23, 1e25, 1e29, 1e31, 1e34, 1e38, 1e200])
@pytest.mark.parametrize("scale", [1e-8, 1e-7, 1e-6, 1e-5, 1e-2, 1.0, 1e3])
def test_screen_skips_only_saturated_indicators(probe, variant, h, scale):
    rng = np.random.default_rng([variant, int(np.log10(h) + 400), int(np.log10(scale) + 50)])
    n = 1500
    rows = np.array([_lines(rng, scale, 10.0 ** rng.uniform(-3, 1)) for _ in range(n)])
    rows[:, 4:] /= h
    a, b = np.zeros((n, 7)), np.zeros((n, 7))
    probe.probe_screen(variant, ctypes.c_double(h), n, *[v.ctypes.data_as(D) for v in (rows, a, b)])
    ok = np.isfinite(b).all(axis=1)
    assert ok.sum() > n // 2
    np.testing.assert_array_equal(a[ok], b[ok])
