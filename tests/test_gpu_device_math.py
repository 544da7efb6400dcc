"""The kernels' own conversions, exp/erfc pair and time coefficients as the GPU
evaluates them: the conversions at their edges, the pair within two ulp and no
further off than the library's functions it replaces, the coefficients rounded
once."""
import ctypes
import os
import subprocess
from decimal import Decimal
from fractions import Fraction

import numpy as np
import pytest

import test_convert_host as conv
import test_gauss_host as gauss
import test_time_coef_ff_host as tc
from paper_2606_17772_gb300 import build as fbuild

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "libdevmath.so")
    subprocess.run([fbuild._nvcc()] + fbuild.NVCC_FLAGS + ["-shared", "-I", fbuild.CSRC, "-o", out,
                   os.path.join(conv.HERE, "device_math_probe.cu"), "-lcudart"], check=True)
    lib = ctypes.CDLL(out)

    def fn(*a):
        assert lib.probe_device(*a) == 0
    return fn


@pytest.mark.filterwarnings("ignore:overflow")
def test_conversions(probe):
    conv.check_conversions(probe)


def test_exp_and_erfc_beat_the_library_pair(probe):
    rng = np.random.default_rng(1)
    k = np.arange(0, 768, 5)
    y = np.concatenate([k / 256.0, (k + 0.5) / 256.0, rng.uniform(0, 3, 600), [0.0, 1e-300, np.nextafter(3.0, 0)]])
    y = np.concatenate([y, -y])
    o = conv.run(probe, 2, y)
    err = np.zeros((len(y), 4))
    for i, v in enumerate(y):
        te, tc_ = gauss._exact(v)
        err[i] = [abs(Decimal(float(a)) - b) / (Decimal(2) ** -52 * b) for a, b in zip(o[i, :4], (te, tc_, te, tc_))]
    assert err[:, :2].max() <= 2.0
    for q in range(2):
        assert err[:, q].max() <= err[:, 2 + q].max() and err[:, q].mean() <= err[:, 2 + q].mean()


def test_time_coefficients_are_rounded_once(probe):
    rng = np.random.default_rng(2)
    n = 300
    dt = 10.0 ** rng.uniform(-6, -1, n)
    tau = dt / 10.0 ** rng.uniform(-6, 0, n)
    tau[:2] = dt[:2]
    o = conv.run(probe, 3, dt, tau)
    for i in range(n):
        for k, r in enumerate(tc._definition(dt[i], tau[i])):
            ulp = Fraction(float(np.spacing(np.float32(abs(float(r))))))
            assert abs(Fraction(o[i, k]) - r) <= (Fraction(1, 2) + Fraction(1, 2048)) * ulp
