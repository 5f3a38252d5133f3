"""End of a step inside the one-launch form of small domains (k_steps): a block
is counted as arrived once all its warps have read the step counter, because
the last block advances it while the others still run.  A warp that reads it
late would trace the wrong step, or find it latched, and meet the block's
barriers out of turn."""
import os
import re

import numpy as np
import pytest

from paper_2207_14496_gb300 import inputs

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2207_14496_gb300", "csrc")


def test_arrival_follows_a_block_barrier():
    """The window is a few instructions wide, so the order is checked in the source:
    the last statement before the arrival, outside every branch that depends
    on the step counter, is a barrier of the block."""
    with open(os.path.join(CSRC, "fsl_kernels.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    body = text[text.index("void end_step_body"):text.index("void __launch_bounds__(256) k_end_step")]
    assert re.search(r"__syncthreads\(\);\s*if \(threadIdx\.x == 0\) last = atomicAdd\(&ctrl->end_blocks",
                     body)


def _wave(L, nz):
    return inputs.standing_wave(L, nz=nz)


def _unstable():
    w = inputs.dam_break(nx=40, ny=40, nz=2, width=12, height=30, g=5e-2, nu=1e-2)
    w["params"]["periodic"] = (False, False, True)
    return w


# trace intervals that divide neither each other nor the steps of a launch, with
# one block, some blocks and a block per SM
@pytest.mark.gpu
@pytest.mark.parametrize("every", [1, 2, 3, 7])
@pytest.mark.parametrize("make,prec", [(lambda: _wave(8, 1), "fp64"), (lambda: _wave(64, 1), "fp64"),
                                       (lambda: _wave(140, 1), "fp64"), (lambda: _wave(200, 2), "fp32"),
                                       (_unstable, "fp64"), (_unstable, "fp16")])
def test_traced_launch_equals_single_steps(fsl, make, prec, every):
    w = make()
    n = 601 if w["phi"].size < 5000 else 301
    got = []
    for parts in ([n], [1] * n):
        sim = fsl.Sim(w["params"], prec)
        sim.init_workload(w)
        sim.set_trace(every)
        for k in parts:
            sim.step(k)
        t = sim.types()
        fl = (t == 1) | (t == 2)
        got.append((sim.trace(n // every), sim.status(), sim.step_count, t, sim.pdfs()[:, fl],
                    sim.phi(), sim.counts(), sim.lost_mass()))
        sim.close()
    for a, b in zip(*got):
        assert np.array_equal(np.asarray(a), np.asarray(b), equal_nan=True)
    assert got[0][1][0] in (0, fsl.ERR_UNSTABLE)
