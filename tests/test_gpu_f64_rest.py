"""The FP64 update where nothing moves (needs a GB300): exact zeros stay exact zeros."""
import numpy as np
import pytest

import oracle
from paper_1810_09299_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("raw", [0, 1])
@pytest.mark.parametrize("nr,nz,zper,lagged", [(33, 40, 0, 0), (64, 64, 1, 1), (97, 130, 0, 0)])
def test_g_of_a_resting_state_stays_zero(nr, nz, zper, lagged, raw):
    """Without surface tension a diffuse drop at rest drives no flow: the oracle's g is zero throughout."""
    case = W.static_drop(nr=nr, nz=nz, R=8.0, sigma=0.0, z_periodic=zper, p_coupling=lagged)
    if raw:
        case = W.with_raw_collision(case)
    phi = W.initial_phi(case)
    assert not oracle.Oracle(case).init(phi).step(5).populations()[1].any()
    sim = lbm.Simulation(case)
    sim.init_phase(0, "host_array", phi=phi)
    sim.step(5)
    assert not sim.state(0)[1].any()
    fields = sim.fields(0)
    assert not any(fields[k].any() for k in ("uz", "ur", "p"))


@pytest.mark.parametrize("raw", [0, 1])
@pytest.mark.parametrize("scale", [1e-250, 1e-285])
def test_vanishing_g_keeps_its_size(scale, raw):
    """g alone, linear in its scale: the smallest values above the unit of the sums (2^-990, 1e-298)
    keep what of them it resolves; 1e-11 of the largest value as in the other FP64 comparisons."""
    case = W.static_drop(nr=33, nz=40, R=8.0, sigma=0.0)
    if raw:
        case = W.with_raw_collision(case)
    rng = np.random.default_rng(1)
    o = oracle.Oracle(case).init(W.initial_phi(case))
    f, g = o.populations()
    g[:] = scale * rng.uniform(-1.0, 1.0, g.shape)
    o.set_populations(f, g)
    sim = lbm.Simulation(case)
    sim.set_state(0, f, g, np.stack(o.aux()))
    o.step(1)
    sim.step(1)
    got, want = sim.state(0)[1], o.populations()[1]
    tol = max(1e-11, 64 * 2.0**-990 / np.max(np.abs(want)))
    assert np.max(np.abs(got - want)) <= tol * np.max(np.abs(want))
