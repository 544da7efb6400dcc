"""The FP32 interface solve does not depend on the density's unit: states scaled
by a power of two in density, at velocities far from 1 too, give the scaled
result wherever FP32 holds it (host build of the kernels' arithmetic)."""
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
    out = str(tmp_path_factory.mktemp("probe") / "libunit.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_2606_17772_gb300", "csrc"), "-o", out,
                    os.path.join(HERE, "host_math_probe.cpp")], check=True)
    return ctypes.CDLL(out)


def solve(probe, base, a, b, mu):
    """Velocities times 2^a, densities times 2^b, the result in the units of base."""
    s = np.array([1.0, 2.0 ** a, 2.0 ** a, 4.0 ** a]) * 2.0 ** b
    inp, out = np.ascontiguousarray(base * np.tile(s, 5)), np.zeros((len(base), 24))
    c = ctypes.c_double
    probe.probe_iface(1, c(1.4), c(mu * 2.0 ** (a + b)), c(1.0), c(0.05), c(1.0), c(0.004 * 2.0 ** -a), 0, len(base),
                      inp.ctypes.data_as(D), out.ctypes.data_as(D))
    return out / np.concatenate([s * 2.0 ** a, s * 4.0 ** a, s, s, s * 2.0 ** a, s * 2.0 ** a])


@pytest.mark.parametrize("mu", [0.0, 0.01])
@pytest.mark.parametrize("a,b", [(0, -100), (0, 29), (0, 30), (0, 31), (0, 100), (-12, 100), (-16, 90), (-20, 100),
                                 (-24, 60), (-24, 100), (12, -100), (14, -100), (16, -90), (18, -85), (18, -100)])
def test_solve_is_linear_in_the_density_unit(probe, a, b, mu):
    rng = np.random.default_rng(0)
    n = 64
    rho, p = rng.uniform(0.5, 2, n), rng.uniform(0.3, 2, n)
    U, V = rng.uniform(-1.5, 1.5, (2, n))
    W = np.stack([rho, rho * U, rho * V, p / 0.4 + 0.5 * rho * (U * U + V * V)], 1)
    base = np.concatenate([W, W * (1 + 0.05 * rng.normal(size=(n, 4)))] +
                          [0.3 * rng.normal(size=(n, 4)) for _ in range(3)], 1)
    ref, out = solve(probe, base, a, 0, mu), solve(probe, base, a, b, mu)
    # powers of two commute with every rounding until a number becomes subnormal; 1e-4 leaves room for those
    assert (np.abs(out - ref).max(0) <= 1e-4 * np.abs(ref).max(0)).all()
