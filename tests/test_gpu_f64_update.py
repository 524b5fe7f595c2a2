"""The FP64 update of the compile-time rate patterns (needs a GB300): edges of
tiles, both collisions and couplings, very small and non-finite values, against
the FP64 oracle.

Tolerance 1e-11 of each output's largest value: a step rounds a few hundred
times at 2^-53, and three steps do not amplify that (the FP64 parity horizon is
ten steps and more).
"""
import numpy as np
import pytest

import oracle
from paper_1810_09299_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-11


def _agree(sim, ref, what=("f", "g", "chi")):
    f, g, aux = sim.state(0)
    rf, rg = ref.populations()
    cz, cr, _ = ref.aux()
    for name, a, b in (("f", f, rf), ("g", g, rg), ("chi", aux[:2], np.stack([cz, cr]))):
        if name in what:
            assert np.max(np.abs(a - b)) <= TOL * np.max(np.abs(b)), name


@pytest.mark.parametrize("raw", [0, 1])
@pytest.mark.parametrize("nr,nz,zper,lagged", [(2, 2, 0, 0), (3, 5, 1, 0), (31, 8, 0, 1), (32, 9, 1, 1), (33, 17, 0, 0),
                                               (64, 16, 1, 0), (65, 34, 0, 0)])
def test_edges_match_oracle(nr, nz, zper, lagged, raw):
    case = W.oscillating_drop(nr=nr, nz=nz, R0=0.3 * nr, ratio=10.0, z_periodic=zper, p_coupling=lagged, grav_z=-1e-5)
    if raw:
        case = W.with_raw_collision(case)
    phi = W.initial_phi(case)
    for v in range(lbm.num_variants()):
        sim = lbm.Simulation(case)
        sim.set_variant(v)
        sim.init_phase(0, "host_array", phi=phi)
        sim.step(3)
        if v == 0:
            first = sim.state(0)
            _agree(sim, oracle.Oracle(case).init(phi).step(3))
        else:  # every launch shape gives the same bits
            for a, b in zip(first, sim.state(0)):
                assert np.array_equal(a, b), v


@pytest.mark.parametrize("raw", [0, 1])
@pytest.mark.parametrize("nz", [3632, 3640, 3645])
def test_many_tiles(nz, raw):
    """33 columns are two tiles per 8 rows: 908, 910 and 912 tiles, the last from six tiles
    per SM on (152 SMs), where another kernel takes over; against 16-row tiles."""
    case = W.oscillating_drop(nr=33, nz=nz, R0=10.0, ratio=10.0)
    if raw:
        case = W.with_raw_collision(case)
    out = []
    for v in (0, 2):
        sim = lbm.Simulation(case)
        sim.set_variant(v)
        sim.init_case(0)
        sim.step(3)
        out.append(sim.state(0))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("raw", [0, 1])
def test_zero_stays_zero(raw):
    """Where phi is exactly zero and nothing moves, f stays exactly zero."""
    case = W.static_drop(nr=64, nz=40, R=8.0, sigma=0.0)
    if raw:
        case = W.with_raw_collision(case)
    phi = W.initial_phi(case)
    phi[phi < 1e-3] = 0.0
    ref = oracle.Oracle(case).init(phi).step(2)
    sim = lbm.Simulation(case)
    sim.init_phase(0, "host_array", phi=phi)
    sim.step(2)
    f, rf = sim.state(0)[0], ref.populations()[0]
    assert (rf == 0).any()
    assert not f[rf == 0].any()


@pytest.mark.parametrize("scale", [1e-40, 1e-200, 1e-270])
def test_very_small_populations(scale):
    """sigma = 0 and f scaled down: phi stays proportional to the scale (n ~ 0 there),
    so the state must keep its relative accuracy."""
    case = W.static_drop(nr=40, nz=48, R=12.0, sigma=0.0)
    phi = W.initial_phi(case)
    ref = oracle.Oracle(case).init(phi * scale).step(2)
    sim = lbm.Simulation(case)
    sim.init_phase(0, "host_array", phi=phi * scale)
    sim.step(2)
    _agree(sim, ref, what=("f",))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e307])
@pytest.mark.parametrize("where", ["f", "g"])
def test_nonfinite_reaches_the_same_nodes(bad, where):
    case = W.static_drop(nr=40, nz=48, R=12.0)
    phi = W.initial_phi(case)
    o = oracle.Oracle(case).init(phi)
    f, g = o.populations()
    (f if where == "f" else g)[5, 20, 11] = bad
    o.set_populations(f, g)
    cz, cr, pp = o.aux()
    sim = lbm.Simulation(case)
    sim.set_state(0, f, g, np.stack([cz, cr, pp]))
    o.step(2)
    sim.step(2)
    a, b = sim.fields(0), o.fields()
    for k in ("phi", "uz", "ur", "p"):
        assert np.array_equal(np.isfinite(a[k]), np.isfinite(b[k])), k
