"""The default bulk variant in domains with free-slip walls, beside which cells
pull direction by direction: about as fast as the plain pair kernel or faster
(the persistent TMA kernel takes up to twice as long there), and the same
bits."""
import numpy as np
import pytest
import torch

from paper_2207_14496_gb300 import inputs

pytestmark = pytest.mark.gpu

# (lattice, shape, periodic axes); the others are free-slip walls
ALL, Y, Z = (False, False, False), (True, False, True), (True, True, False)
CASES = [(19, (150, 150, 150), ALL), (19, (300, 150, 100), (False, False, True)), (27, (150, 150, 150), ALL),
         (27, (400, 400, 20), Z), (19, (400, 400, 20), Z), (19, (200, 200, 100), Y)]


def _run(fsl, w, prec, variant, steps=24):
    sim = fsl.Sim(w["params"], prec)
    sim.set_variant(variant)
    sim.init_workload(w)
    sim.step(steps)
    t = sim.types()
    state = (t, sim.pdfs()[:, (t == 1) | (t == 2)], sim.phi(), sim.status())
    best = np.inf
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(5):
        e0.record(sim.stream)
        sim.step(steps)
        e1.record(sim.stream)
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    sim.close()
    return state, best


@pytest.mark.parametrize("prec", ["fp16", "fp32"])
@pytest.mark.parametrize("q,shape,periodic", CASES)
def test_default_is_no_slower_than_the_pair_kernel(fsl, q, shape, periodic, prec):
    nx, ny, nz = shape
    w = inputs.dam_break(nx=nx, ny=ny, nz=nz, width=nx // 2, height=2 * ny // 3, g=1e-6, nu=1e-2, q=q)
    w["params"].update(periodic=periodic, free_slip=tuple(not p for p in periodic))
    a, ms = _run(fsl, w, prec, "default")
    b, ms_pair = _run(fsl, w, prec, "pair_r128")
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    assert ms < 1.25 * ms_pair
