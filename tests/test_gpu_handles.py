"""Handles that step at the same time, each on its own stream (needs a GB300), share the SMs."""
import time

import pytest

from paper_1810_09299_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "mix_fp16"])
@pytest.mark.parametrize("nr,nz", [(64, 128), (128, 256), (150, 300)])
def test_eight_handles_share_the_sms(nr, nz, prec):
    """Each grid has at most one tile per SM (150 x 300: of 10 rows), and an SM holds the tiles of three
    handles or more: eight handles take two rounds of places, each as long as a step alone or twice
    that, or three rounds."""
    torch = pytest.importorskip("torch")

    def us_per_step(n):
        sims = [lbm.Simulation(W.oscillating_drop(nr=nr, nz=nz, R0=0.25 * nr, precision=prec),
                               stream=torch.cuda.Stream().cuda_stream) for _ in range(n)]
        for s in sims:
            s.init_case(0)
            s.step(64)
        best = float("inf")
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(4):
                for s in sims:
                    s.step(320)
            torch.cuda.synchronize()
            best = min(best, (time.perf_counter() - t) / 1280 * 1e6)
        for s in sims:
            s.close()
        return best

    alone, together = us_per_step(1), us_per_step(8)
    assert together <= 4.0 * alone, (alone, together)
