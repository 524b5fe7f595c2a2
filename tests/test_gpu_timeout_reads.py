"""Reads after a staged step whose bounded wait gave up (needs a GB300): LBM_ERR_TIMEOUT, and the caller's
memory keeps its values, whichever way the read goes."""
import ctypes

import numpy as np
import pytest

from paper_1810_09299_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu
NR, NZ = 96, 96  # five planes are above the size from which pages are touched


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("mask", [1, 31, 3])
def test_fields_are_left_alone(mask, pinned):
    torch = pytest.importorskip("torch")
    sim = lbm.Simulation(W.static_drop(nr=NR, nz=NZ, R=20.0))
    sim.init_case(0)
    sim.step(2)
    buf = torch.full((5 * NR * NZ,), 7.0, dtype=torch.float64, pin_memory=pinned)
    L, dp = lbm.lib(), ctypes.cast(buf.data_ptr(), ctypes.POINTER(ctypes.c_double))
    assert L.lbm_selftest_handle_wait(sim._h, 2000) == lbm.LBM_ERR_TIMEOUT
    assert L.lbm_case_get_fields(sim._h, 0, mask, dp) == lbm.LBM_ERR_TIMEOUT
    assert bool((buf == 7.0).all())
    assert L.lbm_case_get_fields(sim._h, 0, mask, dp) == lbm.LBM_ERR_TIMEOUT  # and stays so


def test_record_and_drops_are_left_alone():
    L = lbm.lib()
    for what in ("record", "drops"):
        sim = lbm.Simulation(W.static_drop(nr=NR, nz=NZ, R=20.0))
        sim.init_case(0)
        assert L.lbm_selftest_handle_wait(sim._h, 2000) == lbm.LBM_ERR_TIMEOUT
        d, drops, n, low = lbm.LbmDiag(step=7.0), (lbm.LbmDrop * 4)(), ctypes.c_int32(7), (ctypes.c_double * 2)(7.0, 7.0)
        drops[0].volume = 7.0
        rc = (L.lbm_case_diagnostics(sim._h, 0, ctypes.byref(d)) if what == "record" else
              L.lbm_case_axis_drops(sim._h, 0, 4, drops, ctypes.byref(n), low))
        assert rc == lbm.LBM_ERR_TIMEOUT
        assert d.step == 7.0 and drops[0].volume == 7.0 and n.value == 7 and list(low) == [7.0, 7.0]


@pytest.mark.parametrize("steps", [3, 70])
def test_staged_steps_read_as_the_others(steps):
    """The TMA-staged variants look at the status word first: same fields."""
    case = W.static_drop(nr=NR, nz=NZ, R=20.0)
    out = []
    for v in (0, 3, 4):
        sim = lbm.Simulation(case)
        sim.set_variant(v)
        sim.init_case(0)
        sim.step(steps)
        out.append([sim.fields(0), sim.fields(0)])
    for a in out:
        for b in a:
            assert all(np.array_equal(b[k], out[0][0][k]) for k in b)
