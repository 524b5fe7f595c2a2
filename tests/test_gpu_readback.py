"""Reads of a running case (needs a GB300): phi alone, the drops on the axis at the edges of
their kernel, and the exact combination of the diagnostics' block sums.
"""
import ctypes
import math

import numpy as np
import pytest

import oracle
from paper_1810_09299_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "mix_fp16", "mix_bf16"])
@pytest.mark.parametrize("nr,nz,raw", [(2, 2, 0), (33, 17, 0), (64, 40, 1), (97, 65, 0)])
def test_phi_alone_is_the_phi_of_all_fields(nr, nz, raw, prec):
    case = W.oscillating_drop(nr=nr, nz=nz, R0=0.3 * nr, ratio=10.0, precision=prec)
    if raw:
        case = W.with_raw_collision(case)
    sim = lbm.Simulation(case)
    sim.init_case(0)
    sim.step(3)
    assert np.array_equal(sim.fields(0, which=("phi",))["phi"], sim.fields(0)["phi"])


@pytest.mark.parametrize("prec", ["fp64", "fp32", "mix_fp16", "mix_bf16"])
@pytest.mark.parametrize("nr,nz", [(2, 2), (33, 17), (97, 65)])
def test_fields_into_page_locked_memory(nr, nz, prec):
    """Stored there by the kernel where the address is aligned, by a copy where it is not or
    where planes are left out: the same values, and nothing beyond them."""
    torch = pytest.importorskip("torch")
    sim = lbm.Simulation(W.oscillating_drop(nr=nr, nz=nz, R0=0.3 * nr, ratio=10.0, precision=prec))
    sim.init_case(0)
    sim.step(2)
    n = nr * nz
    planes = list(sim.fields(0).values())
    for mask in (1, 31, 3, 16):
        want = np.concatenate([planes[i].ravel() for i in range(5) if mask & (1 << i)])
        for offset in (0, 8, 4):
            buf = torch.zeros(8 * (5 * n + 4), dtype=torch.uint8, pin_memory=True)
            rc = lbm.lib().lbm_case_get_fields(sim._h, 0, mask, ctypes.cast(buf.data_ptr() + offset,
                                                                            ctypes.POINTER(ctypes.c_double)))
            assert rc == lbm.LBM_OK
            raw = buf.numpy()
            got = np.frombuffer(raw[offset:offset + 8 * want.size].tobytes())
            assert np.array_equal(got, want)
            assert not raw[:offset].any() and not raw[offset + 8 * want.size:].any()


@pytest.mark.parametrize("zper", [0, 1])
@pytest.mark.parametrize("nz,period", [(2, 2), (3, 3), (255, 7), (256, 2), (257, 16),  # a scan thread's share
                                       (2816, 40), (2817, 40), (5000, 999),            # rows in shared memory, or not
                                       (300, 300), (640, 4)])                          # one run; more than can be stored
def test_axis_drops_at_the_edges(nz, period, zper):
    """Runs of period / 2 liquid rows.  phi differs by 0.8 across a crossing, so positions are
    exact to a few rounding units of nz (1e-11 here) and volumes to the sum's (1e-12 relative,
    33 columns and nz rows)."""
    case = W.static_drop(nr=33, nz=nz, R=1.0, sigma=0.0, z_periodic=zper)
    axis = np.where((np.arange(nz) + period // 4) % period < (period + 1) // 2, 0.9, 0.1)
    phi = axis[:, None] * np.linspace(1.0, 0.2, 33)[None, :]
    phi = np.where(axis[:, None] > 0.5, phi, 0.1)
    sim = lbm.Simulation(case)
    sim.init_phase(0, "host_array", phi=phi)
    got, n, (pmin, zmin) = sim.axis_drops(0)
    ref, n_ref, (pmin_ref, zmin_ref) = oracle.Oracle(case).init(phi).axis_drops()
    assert n == n_ref and len(got) == len(ref)
    assert abs(pmin - pmin_ref) <= 1e-14 and zmin == zmin_ref
    for a, b in zip(got, ref):
        assert abs(a["z_start"] - b["z_start"]) <= 1e-11 and abs(a["z_end"] - b["z_end"]) <= 1e-11
        assert abs(a["volume"] - b["volume"]) <= 1e-12 * abs(b["volume"])


@pytest.mark.parametrize("nz", [2, 31, 33, 255, 256, 257])
@pytest.mark.parametrize("kind", ["plain", "cancelling", "tiny", "huge"])
def test_block_sums_are_added_exactly(nz, kind):
    """One column, one row per block: the mass is the sum of phi / 2 rounded once."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(nz)
    v = rng.uniform(0.1, 1.0, nz) * 10.0 ** rng.integers(-8, 8, nz)
    if kind == "cancelling":
        v[1::2] = -v[0:2 * (nz // 2):2] * (1.0 + rng.uniform(0, 1e-12, nz // 2))
    elif kind == "tiny":
        v *= 2.0 ** -1040
    elif kind == "huge":
        v = rng.uniform(0.1, 1.0, nz) * 2.0 ** 1010
    F = np.zeros((5, nz, 1))
    F[0, :, 0] = v
    d_fields = torch.from_numpy(F).to("cuda")
    d_out = torch.zeros(11, dtype=torch.float64, device="cuda")
    rc = lbm.lib().lbm_diag_reduce_noalloc(ctypes.c_void_p(d_fields.data_ptr()), nz, 1, 0, 0.0,
                                           ctypes.c_void_p(d_out.data_ptr()),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == lbm.LBM_OK
    mass, want = d_out.cpu().numpy()[1], math.fsum(0.5 * x for x in v)
    if kind == "huge":  # beyond the integers' range: plain sums
        assert abs(mass - want) <= nz * 2.0 ** -53 * want
    else:
        assert mass == want
