"""The FP64 reciprocal and square root of the general rates (lbm_device.cuh) against exact quotients and roots
(needs a GB300).

Bounds.  The hardware's starts read and give 32 bits, 20 of them mantissa: e below 2^-19 (measured 2^-19.04 and
2^-19.94 over 2^28 mantissas).  rcp64: the series leaves out e^3.  sqrt64: it leaves out 13/16 e^3.  Both are below
2^-57, 1/16 ulp, before the one rounding: 0.5 + 1/16 + 1/64 ulp.
"""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1810_09299_gb300 import build as B

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    torch = pytest.importorskip("torch")
    out = str(tmp_path_factory.mktemp("rcp64") / "probe.so")
    subprocess.run([B.nvcc(), *B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", out,
                    os.path.join(HERE, "rcp64_probe.cu")], check=True)
    lib = ctypes.CDLL(out)

    def call(root, x):
        t = torch.from_numpy(x).cuda()
        y = torch.empty_like(t)
        torch.cuda.synchronize()
        assert lib.rcp64_run(root, ctypes.c_int64(x.size), ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(y.data_ptr())) == 0
        return y.cpu().numpy()

    return call


def _values():
    rng = np.random.default_rng(3)
    m = np.concatenate([rng.uniform(1.0, 2.0, 200000),
                        1.0 + rng.uniform(0.0, 2.0**-18, 40000), 2.0 - rng.uniform(0.0, 2.0**-18, 40000),
                        1.0 + np.arange(64) * 2.0**-52, 2.0 - np.arange(1, 65) * 2.0**-52,
                        (1.0 + np.arange(1024) / 1024.0) + 2.0**-20 * (1.0 - 2.0**-32)])  # the low word all ones
    return m * 2.0 ** rng.choice([-1, 0, 1, 0, -999, 998, -37, 120], m.size).astype(float)


def _ulps(got, want):
    """|got - want| in ulps of got, want a Fraction."""
    return abs(Fraction(got) - want) / Fraction(float(np.spacing(got)))


@pytest.mark.parametrize("root", [0, 1])
def test_against_the_exact_value(run, root):
    x = _values()
    y = run(root, x)
    near = np.sqrt(x) if root else 1.0 / x  # IEEE, half an ulp
    off = np.abs(y - near) / np.spacing(near)
    assert off.max() <= 1
    # where the two differ, and a few others, against the exact value
    at = np.unique(np.concatenate([np.nonzero(off)[0][:20000], np.arange(0, x.size, 97)]))
    worst = 0
    for i in at:
        v = Fraction(float(x[i]))
        if root:
            s = Fraction(math.isqrt((v.numerator << 400) // v.denominator), 1 << 200)  # to 2^-200
            if v < Fraction(1, 1 << 100):
                s = Fraction(math.isqrt((v.numerator << 2400) // v.denominator), 1 << 1200)
        else:
            s = 1 / v
        worst = max(worst, _ulps(float(y[i]), s))
    print("root" if root else "rcp", "worst %.4f ulp, other than IEEE %.4f" % (float(worst), float((off > 0).mean())))
    assert worst <= Fraction(1, 2) + Fraction(1, 16) + Fraction(1, 64)


def test_ends_of_the_range(run):
    x = np.array([0.0, -0.0, np.inf, np.nan, 5e-324, 2.0**-1022, 2.0**-1074 * 3, 2.0**1023, 1.7976931348623157e308,
                  2.0**-1001, 2.0**-1000, 2.0**1000, 2.0**1001, 2.0**-1030])
    with np.errstate(all="ignore"):
        for root, want in ((0, 1.0 / x), (1, np.sqrt(x))):
            got = run(root, x)
            assert np.array_equal(np.isnan(got), np.isnan(want))
            ok = np.isfinite(want) & (want != 0)
            assert np.array_equal(got[~ok & ~np.isnan(want)], want[~ok & ~np.isnan(want)])
            assert np.all(np.abs(got[ok] - want[ok]) <= np.spacing(want[ok]))
        neg = np.array([-1.0, -2.0**-1020, -np.inf])
        assert np.isnan(run(1, neg)).all()
        assert np.all(np.abs(run(0, -np.abs(_values()[:100])) + 1.0 / np.abs(_values()[:100])) <= np.spacing(1.0 / np.abs(_values()[:100])))
