"""Cell types and bubble labels of small domains are brought into their form on
the host, those of larger ones by a kernel: the same values on both sides of the
bounds, and no slower than a plain field for the smallest domains."""
import time

import numpy as np
import pytest

from paper_2207_14496_gb300 import inputs

pytestmark = pytest.mark.gpu


def _pool(nx, ny):
    w = inputs.bubbles_in_pool(nx=nx, ny=ny, depth=ny - 6, bubbles=((9.0, 9.0, 4.0), (nx - 9.0, 10.0, 4.5)))
    o = np.zeros_like(w["phi"], dtype=np.uint8)
    o[:, 0, ::7] = 1
    w["obstacle"] = o
    return w


# cells: just below and at the bound of the labels (4096), then of the types (65536)
@pytest.mark.parametrize("nx,ny", [(63, 65), (64, 64), (241, 17), (65, 64), (255, 257), (256, 256), (300, 230)])
def test_types_and_labels(fsl, nx, ny):
    w = _pool(nx, ny)
    sim = fsl.Sim(w["params"], "fp32")
    sim.init_workload(w)
    sim.step(6)
    # the same fields from a checkpoint: flags, then labels, in padded rows
    sx, N = (nx + 31) // 32 * 32, (nx + 31) // 32 * 32 * ny
    buf = sim.save()
    plane = (N + 127) // 128 * 128 + 512
    at = 4 * sim.q * plane
    types = buf[at:at + N].reshape(ny, sx)[:, :nx] & 3
    at += N + 4 * 8 * N  # fill level, mass, curvature, lost mass
    lab = buf[at:at + 4 * N].view(np.int32).reshape(ny, sx)[:, :nx]
    want = np.where(lab >= 0, lab % sx + nx * (lab // sx), lab)
    got_t, got_l = sim.types()[0], sim.bubbles()[0]
    assert np.array_equal(got_t, types) and set(np.unique(got_t)) == {0, 1, 2, 3}
    assert np.array_equal(got_l, want) and got_l.max() >= 0
    sim.close()


def test_small_domains(fsl):
    w = inputs.standing_wave(64)
    sim = fsl.Sim(w["params"], "fp32")
    sim.init_workload(w)
    sim.step(2)
    t, f = np.zeros(sim.N, np.uint8), np.zeros(sim.N)

    def best(what, out, n=1500):
        b = np.inf
        for _ in range(n):
            a = time.perf_counter()
            sim._obs(what, out)
            b = min(b, time.perf_counter() - a)
        return b

    for _ in range(6):  # a busy host may spoil some of the tries
        if best(fsl.OBS_FIELD_TYPES, t) < 1.12 * best(fsl.OBS_FIELD_PHI, f):
            break
    else:
        raise AssertionError("cell types take longer than the fill level")
    sim.close()
