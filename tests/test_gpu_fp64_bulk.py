"""The FP64 bulk pass against the oracle, bit for bit, where its collision
changes form: the additions near 1 run in fixed point while |u|^2 < 0.015 and
as FP64 additions above, and operands may be zero, tiny or exact ties."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _box(shape, q, collision, g, seed, scale):
    nx, ny, nz = shape
    r = np.random.default_rng(seed)
    u = r.uniform(-1.0, 1.0, (nz, ny, nx, 3))
    u *= scale / np.linalg.norm(u, axis=-1, keepdims=True) * r.uniform(0.0, 1.0, (nz, ny, nx, 1))
    k = r.integers(0, 6, (nz, ny, nx))
    u[k == 0] = 0.0
    u[k == 1] *= 2.0 ** -r.integers(20, 60, (int((k == 1).sum()), 1)).astype(float)
    # few significant bits: sums and products that tie
    u[k == 2] = np.round(u[k == 2] * 64) / 64
    params = dict(q=q, collision=collision, magic=3.0 / 16.0, refill="eq", shape=shape,
                  periodic=(True, False, True), nu=0.02, g=g, sigma=0.0, p_v=1.0 / 3.0, eps=1e-2,
                  options=0)
    return params, np.ones((nz, ny, nx)), u


# nx: one cell, the last lane of a warp, one past it, two blocks and a bit
@pytest.mark.parametrize("nx", [1, 31, 33, 70])
@pytest.mark.parametrize("q,collision,g", [(19, "srt", (0.0, -1e-5, 0.0)), (27, "trt", (0.0, 0.0, -1e-6)),
                                           (27, "srt", (1e-6, 0.0, 0.0)), (19, "trt", (1e-6, -2e-6, 0.0)),
                                           (27, "trt", (0.0, 0.0, 0.0))])
@pytest.mark.parametrize("scale", [0.08, 0.17])
def test_fp64_collision_bits(fsl, nx, q, collision, g, scale):
    """A liquid box whose velocities reach below and above |u| = sqrt(0.015):
    PDFs equal the oracle's exactly (no rounding may differ) after 3 steps."""
    params, phi, u0 = _box((nx, 6, 4), q, collision, g, 17 * nx + q, scale)
    sim, orc = fsl.Sim(params, "fp64"), oracle.Oracle(params)
    sim.init_fill(phi, u0)
    orc.init_fill(phi, u0)
    for step in range(3):
        sim.step(1)
        orc.step(1)
        assert np.array_equal(sim.pdfs(), orc.pdfs()), f"step {step + 1}"
    assert sim.status()[0] == 0
