"""The table-driven exp(-y^2) and erfc(y) of the FP64 half-space moments
against 50-digit values: at the table's points, half-way between them (the
ends of each expansion), beyond the table and at random."""
import ctypes
import os
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))
PI = Decimal("3.14159265358979323846264338327950288419716939937510582097494459")


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "libgauss.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_2606_17772_gb300", "csrc"), "-o", out,
                    os.path.join(HERE, "gauss_probe.cpp")], check=True)
    return ctypes.CDLL(out)


def _exact(y):
    getcontext().prec = 60
    y = Decimal(float(y))
    term, s, n = y, y, 0
    while abs(term) > Decimal(10) ** -55:
        n += 1
        term = -term * y * y / n
        s += term / (2 * n + 1)
    return (-y * y).exp(), 1 - 2 * s / PI.sqrt()


def test_pair_within_two_ulp(probe):
    rng = np.random.default_rng(0)
    k = np.concatenate([np.arange(0, 768, 7), [1, 2, 765, 766, 767]])
    y = np.concatenate([k / 256.0, (k + 0.5) / 256.0, np.nextafter((k + 0.5) / 256.0, 0), rng.uniform(0, 3, 400),
                        [0.0, 1e-300, 1e-9, np.nextafter(3.0, 0), 3.0, 3.5, 4.0]])
    y = np.concatenate([y, -y])
    e, ec = np.zeros_like(y), np.zeros_like(y)
    D = ctypes.POINTER(ctypes.c_double)
    probe.probe_exp_erfc(len(y), y.ctypes.data_as(D), e.ctypes.data_as(D), ec.ctypes.data_as(D))
    ulp = Decimal(2) ** -52
    for a, b, c in zip(y, e, ec):
        te, tc = _exact(a)
        # table entry and final sum half an ulp each, the expansion (at most 1.2 % of the value) the rest; beyond
        # the table the library's functions, whose argument -y^2 is rounded (y^2/2 ulp)
        tol = (Decimal(2) if abs(a) < 3 else Decimal(10)) * ulp
        assert abs(Decimal(float(b)) - te) <= tol * te, a
        assert abs(Decimal(float(c)) - tc) <= tol * tc, a
