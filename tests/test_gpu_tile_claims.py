"""The TMA bulk kernel hands out the tiles of narrow domains by a counter once
every block's ring has been filled: with more tiles than blocks times ring
stages (and with fewer tiles than blocks) every tile is updated exactly once,
so the state equals the pair kernel's bit for bit."""
import numpy as np
import pytest

from paper_2207_14496_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("q,shape", [(19, (30, 41, 700)), (19, (64, 5, 1901)), (27, (33, 17, 600)),
                                     (19, (30, 7, 3)), (27, (100, 3, 1000))])
def test_claimed_tiles_equal_pair(fsl, q, shape, prec):
    nx, ny, nz = shape
    w = inputs.dam_break(nx=nx, ny=ny, nz=nz, width=nx - 3, height=ny - 2, g=1e-4, nu=1e-2, q=q)
    got = []
    for variant in ("pair", "tma"):
        sim = fsl.Sim(w["params"], prec)
        sim.set_variant(variant)
        sim.init_workload(w)
        sim.step(1)
        sim.step(6)
        t = sim.types()
        got.append((t, sim.pdfs()[:, (t == 1) | (t == 2)], sim.phi(), sim.status()))
        sim.close()
    assert got[0][3][0] == 0
    for a, b in zip(got[0], got[1]):
        assert np.array_equal(a, b)
