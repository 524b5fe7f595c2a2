"""The combination of the diagnostics' block sums where large ones cancel (needs a GB300): what is left keeps
its accuracy, however far below them it lies."""
import ctypes
import math

import numpy as np
import pytest

from paper_1810_09299_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [3, 33, 65, 257])
@pytest.mark.parametrize("low", [1e-12, 1e-25, 1e-40, 1e-150, 1e-295])
def test_what_cancellation_leaves(nz, low):
    """One column, one row per block: the mass is the sum of phi / 2.  Pairs that cancel exactly, of sizes up to
    2^200 apart, around values of the size `low`.  The windows' sums are exact and added with compensation: two
    units in the last place."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(nz)
    n = nz // 3
    big = rng.uniform(0.5, 1.0, n) * 2.0 ** rng.integers(-100, 100, n)
    v = np.concatenate([big, -big, low * rng.uniform(0.5, 1.0, nz - 2 * n)])
    rng.shuffle(v)
    F = np.zeros((5, nz, 1))
    F[0, :, 0] = v
    d_fields = torch.from_numpy(F).to("cuda")
    d_out = torch.zeros(11, dtype=torch.float64, device="cuda")
    rc = lbm.lib().lbm_diag_reduce_noalloc(ctypes.c_void_p(d_fields.data_ptr()), nz, 1, 0, 0.0,
                                           ctypes.c_void_p(d_out.data_ptr()),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == lbm.LBM_OK
    mass, want = d_out.cpu().numpy()[1], math.fsum(0.5 * x for x in v)
    assert want > 0 and abs(mass - want) <= 2 * np.spacing(want), (mass, want)
