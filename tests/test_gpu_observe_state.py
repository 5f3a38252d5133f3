"""Observing a simulation leaves its state alone: a checkpoint taken later holds
the same bytes (those of gas and obstacle cells and of the padding among them)
whether fields were read in between or not."""
import numpy as np
import pytest

from paper_2207_14496_gb300 import inputs

pytestmark = pytest.mark.gpu


def _obstacle():
    w = inputs.dam_break(nx=41, ny=33, nz=5, width=15, height=20, g=1e-4, nu=1e-2, refill="geq")
    o = np.zeros_like(w["phi"], dtype=np.uint8)
    o[:, 0:5, 20:27] = 1
    w["obstacle"] = o
    return w


def _bubbles():
    return inputs.bubbles_in_pool(nx=40, ny=24, depth=18, bubbles=((10.0, 8.0, 4.0), (28.0, 9.0, 4.5)))


# rows padded (41, 40) and not (64), one cell wide (a scratch of many planes)
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("make", [_obstacle, _bubbles, lambda: inputs.standing_wave(64, nz=2, q=27),
                                  lambda: inputs.dam_break(nx=1, ny=20, nz=3, width=1, height=9,
                                                           g=1e-4, nu=1e-2)])
def test_observation_leaves_the_state(fsl, make, prec):
    w = make()
    sim = fsl.Sim(w["params"], prec)
    sim.init_workload(w)
    sim.step(7)
    start = sim.save()
    saved, fields = [], []
    for look in (False, True):
        for n in (1, 4):
            # both PDF buffers as a run of known length leaves them
            sim.load(start)
            sim.step(13)
            sim.load(start)
            for _ in range(3):
                if look:
                    fields.append([sim.pdfs(), sim.types(), sim.bubbles(), sim.phi(), sim.pressure(),
                                   sim.total_mass(), sim.max_velocity()])
                sim.step(n)
            saved.append(sim.save())
    assert np.array_equal(saved[0], saved[2]) and np.array_equal(saved[1], saved[3])
    # the fields of the loaded state, read twice: the same values
    for a, b in zip(fields[0], fields[3]):
        assert np.array_equal(a, b, equal_nan=True)
    if prec == "fp64":
        # every plane, non-fluid cells too, as the checkpoint holds it
        (nx, ny, nz), q = sim.shape, sim.q
        sx = (nx + 31) // 32 * 32
        plane = (sx * ny * nz + 127) // 128 * 128 + 512
        raw = start[:8 * q * plane].view(np.float64).reshape(q, plane)[:, :sx * ny * nz]
        raw = raw.reshape(q, nz, ny, sx)[..., :nx]
        assert np.array_equal(fields[0][0], raw, equal_nan=True)
    sim.close()
