"""The 62-bit numbers of the FP64 update (lbm_fix64.cuh), one operation at a time against whole
numbers: on the host with FP32 starts one ulp off either way, and on the GPU with its own starts.

Bounds: a product leaves out -2 to 14 units and adds 4 back: within 10.  rcp and root keep less than 8 units of their last
place of 2^-61 or better: within 2^-58 of themselves.  Quotients by 3 and 9 within 1.5 units.
"""
import ctypes
import os
import random
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
MUL, RCP, ROOT, THIRD, NINTH = range(5)
TOP = 1 << 62


def _compile(cmd, where):
    out = os.path.join(where, "fix64_probe.so")
    subprocess.run([*cmd, "-o", out, os.path.join(HERE, "fix64_probe.cu")], check=True)
    return ctypes.CDLL(out)


@pytest.fixture(scope="module", params=[-1, 0, 1])
def host(request, tmp_path_factory):
    """run(op, a, b) on the host; a and b are lists of (m, e)."""
    cxx = shutil.which("g++") or shutil.which("c++")
    lib = _compile([cxx, "-x", "c++", "-std=c++17", "-O2", "-ffp-contract=off", "-fwrapv", "-w", "-shared", "-fPIC"],
                   str(tmp_path_factory.mktemp("fix64")))
    lib.fix64_start_ulps(request.param)

    def run(op, a, b):
        am, ae, bm, be, rm, re = _arrays(a, b)
        p = lambda x: ctypes.c_void_p(x.ctypes.data)  # noqa: E731
        assert lib.fix64_run(op, ctypes.c_int64(len(a)), p(am), p(ae), p(bm), p(be), p(rm), p(re)) == 0
        return list(zip(rm.tolist(), re.tolist()))

    return run


@pytest.fixture(scope="module")
def gpu(tmp_path_factory):
    torch = pytest.importorskip("torch")
    from paper_1810_09299_gb300 import build as B
    lib = _compile([B.nvcc(), *B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC"],
                   str(tmp_path_factory.mktemp("fix64")))

    def run(op, a, b):
        t = [torch.from_numpy(x).cuda() for x in _arrays(a, b)]
        torch.cuda.synchronize()
        assert lib.fix64_run(op, ctypes.c_int64(len(a)), *(ctypes.c_void_p(x.data_ptr()) for x in t)) == 0
        return list(zip(t[4].tolist(), t[5].tolist()))

    return run


def _arrays(a, b):
    col = lambda v, i, t: np.array([x[i] for x in v], dtype=t)  # noqa: E731
    n = len(a)
    return (col(a, 0, np.int64), col(a, 1, np.int32), col(b, 0, np.int64), col(b, 1, np.int32), np.zeros(n, np.int64),
            np.zeros(n, np.int32))


def _positive():
    """Around the powers of two, just below 1 (where the FP32 start decides), and anywhere."""
    rng = random.Random(5)
    v = [TOP - (1 << (62 - k)) for k in range(2, 63)] + [(TOP >> 1) + (1 << (61 - k)) for k in range(1, 62)]
    v += [TOP >> 1, 1, 2, 3]
    v += [576460696692673444]  # 1 - 9.65e-8 in units of 2^-59
    v += [int(TOP * (1.0 - rng.uniform(0.0, 6e-7))) - rng.randrange(512) for _ in range(4000)]
    v += [int((TOP >> 1) * (1.0 + rng.uniform(0.0, 6e-7))) + rng.randrange(512) for _ in range(4000)]
    v += [rng.randrange(TOP >> 1, TOP) for _ in range(4000)]
    v += [rng.randrange(1, 1 << rng.randrange(1, 62)) for _ in range(1000)]
    return [(m, e) for m in v for e in (-62, -61, -62 + rng.randrange(-900, 900))]


def _check_rcp(run):
    a = [(s * m, e) for m, e in _positive() for s in (1, -1)]
    for (m, e), (rm, re) in zip(a, run(RCP, a, a)):
        # |r a - 1| <= 2^-58
        k = -(re + e)
        assert k >= 0 and abs(rm * m - (1 << k)) << 58 <= 1 << k, (m, e)
        assert abs(rm) < TOP


def _check_root(run):
    a = _positive()
    for (m, e), (rm, re) in zip(a, run(ROOT, a, a)):
        # |r^2 / a - 1| <= 2^-57 (twice the bound of the root), and the root fits a factor
        k = e - 2 * re
        assert k >= 0 and abs(rm * rm - (m << k)) << 57 <= m << k, (m, e)
        assert 0 < rm < TOP
    (zero,) = run(ROOT, [(0, -5)], [(0, 0)])
    assert zero[0] == 0


def _check_mul(run):
    rng = random.Random(6)
    ends = [TOP - 1, TOP - 2, TOP >> 1, (TOP >> 1) + 1, (TOP >> 1) - 1, (1 << 32) - 1, 1 << 32, 1 << 31, 1, 0]
    ends += [-x for x in ends] + [-TOP]
    pairs = [(x, y) for x in ends for y in ends if (x, y) != (-TOP, -TOP)]
    pairs += [(rng.randrange(-TOP, TOP), rng.randrange(-TOP, TOP)) for _ in range(20000)]
    a, b = [(x, 3) for x, _ in pairs], [(y, -7) for _, y in pairs]
    for (x, y), (rm, re) in zip(pairs, run(MUL, a, b)):
        assert re == 58 and abs((rm << 62) - x * y) <= 10 << 62, (x, y)


def _check_quotients(run):
    rng = random.Random(7)
    v = [0, 1, -1, 2, -2, 8, 9, -9, TOP, -TOP, 2 * TOP - 1, -2 * TOP, (1 << 32) - 1, 1 << 32, -(1 << 32)]
    v += [rng.randrange(-2 * TOP, 2 * TOP) for _ in range(20000)]
    a = [(x, 0) for x in v]
    for op, d in ((THIRD, 3), (NINTH, 9)):
        for x, (rm, _) in zip(v, run(op, a, a)):
            assert 2 * abs(d * rm - x) <= 3 * d, (d, x)


@pytest.mark.parametrize("check", [_check_rcp, _check_root, _check_mul, _check_quotients])
def test_operations_on_the_host(host, check):
    check(host)


@pytest.mark.gpu
@pytest.mark.parametrize("check", [_check_rcp, _check_root, _check_mul, _check_quotients])
def test_operations_on_the_gpu(gpu, check):
    check(gpu)
