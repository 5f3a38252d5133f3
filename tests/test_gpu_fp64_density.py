"""The density sum of the FP64 bulk pass, bit for bit against the oracle, at the
ends of the range that its fixed-point form covers: partial sums that come to
1/4 or 2 from either side within fractions of their last place, through
negative PDFs, and the binade borders 1/2 and 1 between them."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SHAPE = (96, 16, 8)


def _columns(q, seed):
    """One PDF vector per cell.  f_0 .. f_3 bring the partial sum to a border b
    give or take fractions of its last place; the others are equal numbers of
    few bits, opposite directions alike, that keep the difference visible."""
    r = np.random.default_rng(seed)
    n = int(np.prod(SHAPE))
    b = r.choice([0.25, 0.25, 0.5, 1.0, 2.0], n)
    ulp = b * 2.0 ** -52
    f = np.zeros((q, n))
    f[0] = np.where(b == 2.0, 0.9, np.where(b == 1.0, 0.5, b)) + r.integers(0, 9, n) * ulp / 2
    gap = b - f[0]
    back = r.integers(-40, 41, n) * ulp / r.choice([1.0, 2.0, 64.0, 128.0], n)
    # the larger gaps in two halves of opposite directions (no velocity of 1)
    f[1] = np.where(b >= 1.0, gap / 2, gap) + back
    f[2] = np.where(b >= 1.0, gap / 2, 0.0) + r.integers(-8, 300, n) * ulp / r.choice([8.0, 64.0], n)
    f[3] = r.choice([0.0, -0.0, 1.0, -1.0, 0.75], n) * ulp / r.choice([1.0, 2.0, 4.0], n)
    # 1/4 - 2^-55 is an FP64 number, which rounding to multiples of 2^-54 loses
    f[:4, :64] = np.array([0.25 + 2.0 ** -54, -(2.0 ** -54 + 20 * 2.0 ** -60), 3 * 2.0 ** -56, 0.0])[:, None]
    f[5:] = (r.integers(0, 3, n) * 2.0 ** -10) * np.where(b == 2.0, 0.0, 1.0)
    return f


@pytest.mark.parametrize("q,collision,g", [(19, "srt", (0.0, 0.0, 0.0)), (19, "trt", (0.0, -1e-5, 0.0)),
                                           (27, "srt", (1e-6, -2e-6, 0.0)), (27, "trt", (0.0, 0.0, -1e-6))])
def test_density_at_the_range_ends(fsl, q, collision, g):
    nx, ny, nz = SHAPE
    params = dict(q=q, collision=collision, magic=3.0 / 16.0, refill="eq", shape=SHAPE,
                  periodic=(True, True, True), nu=0.02, g=g, sigma=0.0, p_v=1.0 / 3.0, eps=1e-2, options=0)
    phi = np.ones((nz, ny, nx))
    sim, orc = fsl.Sim(params, "fp64"), oracle.Oracle(params)
    sim.init_fill(phi)
    orc.init_fill(phi)
    want = _columns(q, 5 + q).reshape(q, nz, ny, nx)
    # cell x pulls f_i from x - c_i
    c, _, _ = orc.lattice()
    stored = np.stack([np.roll(want[i], (-c[i][2], -c[i][1], -c[i][0]), (0, 1, 2)) for i in range(q)])
    state = sim.save()
    plane = nx * ny * nz + 512  # (rows are a multiple of 32, the domain of 128 cells)
    state[:8 * q * plane].view(np.float64).reshape(q, plane)[:, :nx * ny * nz] = stored.reshape(q, -1)
    sim.load(state)
    assert np.array_equal(sim.pdfs(), stored)
    orc.set_state(orc.types(), phi, stored)
    sim.step(1)
    orc.step(1)
    assert sim.status()[0] == 0
    assert np.array_equal(sim.pdfs(), orc.pdfs())
    sim.close()
