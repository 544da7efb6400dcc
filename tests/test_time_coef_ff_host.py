"""The mixed path's time coefficients for dt/tau <= 1 carry no more error than
the FP64 form rounded to FP32 would: each is the definition's value (App. A1's
fit to the time integrals of f, in exact fractions) rounded once."""
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
    out = str(tmp_path_factory.mktemp("probe") / "libtcff.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_2606_17772_gb300", "csrc"), "-o", out,
                    os.path.join(HERE, "time_coef_ff_probe.cpp")], check=True)
    return ctypes.CDLL(out)


def _definition(dt, tau):
    dt, tau = Fraction(float(dt)), Fraction(float(tau))

    def integrals(d):
        y = Fraction(int(d / tau * 2 ** 220), 2 ** 220)
        term, em = Fraction(1), Fraction(0)
        for n in range(1, 36):                # 1/36! < 2^-138
            term = Fraction(int(-term * y / n * 2 ** 300), 2 ** 300)
            em += term                        # exp(-y) - 1
        e1, E = -em, 1 + em
        return (d - tau * e1, -tau * d * (1 + E) + 2 * tau * tau * e1, d * d / 2 - tau * d + tau * tau * e1), E
    Ch, _ = integrals(dt / 2)
    Cf, E = integrals(dt)
    cn = [(4 * h - f) / dt for h, f in zip(Ch, Cf)]
    ct = [4 * (f - 2 * h) / (dt * dt) for h, f in zip(Ch, Cf)]
    cn += [1 - cn[0], -tau - cn[1], -tau - cn[2]]
    ct += [-ct[0], -ct[1], 1 - ct[2]]
    return cn + ct + [E, 1 - E]


@pytest.mark.parametrize("lo,hi", [(-6, -3), (-3, -1), (-1, 0)])
def test_coefficients_are_rounded_once(probe, lo, hi):
    rng = np.random.default_rng(lo + 10)
    n = 200
    dt = 10.0 ** rng.uniform(-6, -1, n)
    tau = dt / 10.0 ** rng.uniform(lo, hi, n)
    if hi == 0:
        tau[:2] = dt[:2]
    a, b = np.zeros((n, 14)), np.zeros((n, 14))
    D = ctypes.POINTER(ctypes.c_double)
    probe.probe_time_coef(n, *[v.ctypes.data_as(D) for v in (dt, tau, a, b)])
    ea, eb = np.zeros((n, 14)), np.zeros((n, 14))
    for i in range(n):
        for k, r in enumerate(_definition(dt[i], tau[i])):
            ulp = Fraction(float(np.spacing(np.float32(abs(float(r))))))
            ea[i, k] = abs(Fraction(a[i, k]) - r) / ulp
            eb[i, k] = abs(Fraction(b[i, k]) - r) / ulp
    # one rounding is half an ulp; the series' own error is below 2^-38, 2^-14 of an ulp, three times that where
    # the terms of a sum cancel
    assert ea.max() <= 0.5 + 2.0 ** -11
    assert ea.max() <= eb.max() + 2.0 ** -11
