"""The conversions by shifts (est_f32, f32_to_f64) at their edges, in the form
that the GPU runs too."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))
D = ctypes.POINTER(ctypes.c_double)


def values(rng):
    """FP64 values around every edge of FP32, and over its whole range."""
    edge = np.array([2.0 ** k for k in (-1074, -1022, -150, -149, -127, -126, -125, -1, 0, 1, 127, 128, 129, 1023)])
    x = np.concatenate([edge, np.nextafter(edge, 0), np.nextafter(edge, np.inf), edge * (1 + 2.0 ** -24),
                        edge * (1 + 2.0 ** -23), rng.normal(size=2000) * 10.0 ** rng.uniform(-46, 40, 2000),
                        [0.0, 1.0 / 3, np.inf]])
    return np.concatenate([x, -x])


def truncated(x):
    """x cut to 24 bits, zero below 2^-126, infinite from 2^128 on."""
    m, e = np.frexp(x)
    t = np.ldexp(np.trunc(np.ldexp(m, 24)), e - 24)
    t = np.where(np.abs(x) < 2.0 ** -126, 0.0, t)
    return np.copysign(np.where(np.abs(x) >= 2.0 ** 128, np.inf, t), x)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "libconv.so")
    subprocess.run(["g++", "-x", "c++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_2606_17772_gb300", "csrc"), "-o", out,
                    os.path.join(HERE, "device_math_probe.cu")], check=True)
    return ctypes.CDLL(out)


def run(fn, what, x, y=None):
    x = np.ascontiguousarray(x, dtype=np.float64)
    y = np.zeros_like(x) if y is None else np.ascontiguousarray(y, dtype=np.float64)
    out = np.zeros((len(x), 14))
    fn(what, len(x), *[a.ctypes.data_as(D) for a in (x, y, out)])
    return out


def check_conversions(fn):
    x = values(np.random.default_rng(0))
    est = run(fn, 0, x)[:, 0]
    np.testing.assert_array_equal(est, truncated(x))
    np.testing.assert_array_equal(np.signbit(est), np.signbit(x))
    assert np.isinf(run(fn, 0, [np.nan])[0, 0])
    back = run(fn, 1, x)[:, 0]
    f = x.astype(np.float32).astype(np.float64)
    normal = np.isfinite(f) & (np.abs(f) >= 2.0 ** -126)
    np.testing.assert_array_equal(back[normal], f[normal])
    small = np.abs(f) < 2.0 ** -126
    assert (np.abs(back[small] - f[small]) <= 2.0 ** -127).all()


@pytest.mark.filterwarnings("ignore:overflow")
def test_conversions(probe):
    check_conversions(probe.probe_host)
