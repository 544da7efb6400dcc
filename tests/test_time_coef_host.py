"""The FP32 path's series of the interface distribution's time coefficients
for dt/tau <= 1 against their definition (the fit of App. A1 to the time
integrals of f), evaluated with 40 digits: the definition's terms cancel to
third order in dt/tau, which FP64 itself loses below dt/tau = 1e-3."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "libtc.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_2606_17772_gb300", "csrc"), "-o", out,
                    os.path.join(HERE, "time_coef_probe.cpp")], check=True)
    return ctypes.CDLL(out)


def _definition(dt, tau):
    """cn[6], ct[6], E, 1 - E in exact fractions (exp by 40 terms, |x| <= 1)."""
    dt, tau = Fraction(float(dt)), Fraction(float(tau))

    def integrals(d):
        y, term, em = d / tau, Fraction(1), Fraction(0)
        for n in range(1, 40):
            term = -term * y / n
            em += term                        # exp(-y) - 1
        e1, E = -em, 1 + em
        return (d - tau * e1, -tau * d * (1 + E) + 2 * tau * tau * e1, d * d / 2 - tau * d + tau * tau * e1), E
    Ch, _ = integrals(dt / 2)
    Cf, E = integrals(dt)
    cn = [(4 * h - f) / dt for h, f in zip(Ch, Cf)]
    ct = [4 * (f - 2 * h) / (dt * dt) for h, f in zip(Ch, Cf)]
    cn += [1 - cn[0], -tau - cn[1], -tau - cn[2]]
    ct += [-ct[0], -ct[1], 1 - ct[2]]
    return [float(v) for v in cn + ct + [E, 1 - E]]


def test_series_match_the_definition(probe):
    rng = np.random.default_rng(0)
    n = 150
    dt = (10.0 ** rng.uniform(-6, -1, n)).astype(np.float32)
    x = 10.0 ** rng.uniform(-6, 0, n)
    x[:3] = 1.0, 1e-6, 0.999
    tau = np.maximum(dt / x, dt).astype(np.float32)
    out = np.zeros((n, 14))
    F, D = ctypes.POINTER(ctypes.c_float), ctypes.POINTER(ctypes.c_double)
    probe.probe_time_coef_small(n, dt.ctypes.data_as(F), tau.ctypes.data_as(F), out.ctypes.data_as(D))
    ref = np.array([_definition(a, b) for a, b in zip(dt, tau)])
    # Horner's leading term (half an ulp and as much again from the rest, up to a factor of 2 where the alternating
    # terms cancel at x = 1), x itself (half an ulp, up to squared), two products: 8 ulp
    assert np.max(np.abs(out - ref) / np.abs(ref)) < 8 * 2.0 ** -23
