"""Variant 0's tile height (needs a GB300): on grids of a little more than one or two 8-row
tiles per SM (152) the same kernel runs tiles of 10 or 12 rows.  Every result is that of the
4-row tiles (variant 2), bit for bit, in every precision and collision.
"""
import numpy as np
import pytest

from paper_1810_09299_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "mix_fp16", "mix_bf16"])
@pytest.mark.parametrize("coll", ["paper", "raw", "general"])
@pytest.mark.parametrize("nr,nz", [(33, 608),    # 152 tiles of 8 rows: 8
                                   (33, 609),    # 154; 122 of 10: 10
                                   (64, 760),    # 152 of 10
                                   (64, 761),    # 154 of 10; 128 of 12: 12
                                   (101, 333),   # 10, a ragged last tile and column
                                   (65, 601),    # 12, one row in the last tile
                                   (200, 400)])  # two CTAs of 10 rows per SM (FP64: 8)
def test_matches_four_row_tiles(nr, nz, coll, prec):
    case = W.oscillating_drop(nr=nr, nz=nz, R0=10.0, ratio=10.0, z_periodic=int(nr == 64), precision=prec)
    if coll == "raw":
        case = W.with_raw_collision(case)
    if coll == "general":
        case["sg"] = [1.0, -1.0, 0.9, 1.1, 1.2, 1.05, 0.95, -1.0, -1.0]
    out = []
    for v in (0, 2):
        sim = lbm.Simulation(case)
        sim.set_variant(v)
        sim.init_case(0)
        sim.step(35)
        out.append(sim.state(0))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", ["fp32", "mix_fp16"])
@pytest.mark.parametrize("nr,nz", [(33, 40), (64, 152), (128, 256), (150, 400), (200, 400)])
def test_early_launches_beside_reads_and_another_stream(nr, nz, prec):
    """Up to two tiles per SM the next step's blocks are launched while a step runs: steps by
    graph and one by one, reads between them and a second handle on its own stream."""
    torch = pytest.importorskip("torch")
    case = W.oscillating_drop(nr=nr, nz=nz, R0=10.0, ratio=10.0, precision=prec)
    ref = lbm.Simulation(case)
    ref.set_variant(2)
    ref.init_case(0)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    sims = [lbm.Simulation(case, stream=s.cuda_stream) for s in streams]
    for s in sims:
        s.set_variant(0)
        s.init_case(0)
    for n in (1, 2, 33, 64, 5):
        ref.step(n)
        for s in sims:
            s.step(n)
        want = ref.fields(0)
        for s in sims:
            got = s.fields(0)
            assert all(np.array_equal(got[k], want[k]) for k in want)
            s.diagnostics(0)
    for s in sims:
        for a, b in zip(s.state(0), ref.state(0)):
            assert np.array_equal(a, b)
