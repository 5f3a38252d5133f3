"""Small domains advance many steps in one launch (k_steps); single steps take
the separate launches.  Both run the same phases, so every field, the trace,
the counters and the instability latch must agree bit for bit."""
import numpy as np
import pytest

from paper_2207_14496_gb300 import inputs

pytestmark = pytest.mark.gpu


def _freeslip():
    w = inputs.dam_break(nx=90, ny=50, nz=1, width=20, height=30, g=2e-4, nu=2e-3, refill="avg")
    w["params"].update(periodic=(False, False, True), free_slip=(True, True, False), les_cs=0.1,
                       sigma=1e-5)
    return w


def _obstacle():
    w = inputs.dam_break(nx=70, ny=40, nz=3, width=20, height=26, g=2e-4, nu=5e-3, refill="ext")
    o = np.zeros_like(w["phi"], dtype=np.uint8)
    o[:, 0:6, 34:40] = 1
    w["obstacle"] = o
    return w


def _unstable():
    w = inputs.dam_break(nx=40, ny=40, nz=1, width=12, height=30, g=5e-2, nu=1e-2)
    w["params"]["periodic"] = (False, False, True)
    return w


def _narrow():
    return inputs.dam_break(nx=3, ny=20, nz=2, width=2, height=10, g=1e-4, nu=1e-2, refill="eq_neq")


CASES = {
    "wave33": (lambda: inputs.standing_wave(33, nz=2, refill="geq"), ("fp64", "fp32", "fp16")),
    "freeslip_les": (_freeslip, ("fp64", "fp32", "bf16")),
    "obstacle": (_obstacle, ("fp64", "fp32", "fp16")),
    "drop27": (lambda: inputs.drop_impact(n=32, pool=10, diameter=10.0, gap=8.0, speed=0.05,
                                          sigma=1e-3, g=1e-5, nu=5e-3, nxy=30), ("fp32", "fp16")),
    "force_x": (lambda: inputs.poiseuille(ny=20, nx=40), ("fp64", "fp32")),
    "narrow": (_narrow, ("fp64", "fp16")),
    "unstable": (_unstable, ("fp64", "fp32")),
    # the most cells a block per SM is given
    "wave440": (lambda: inputs.standing_wave(440, nz=1, nu=1e-3), ("fp16",)),
}


def _state(sim, n):
    t = sim.types()
    fl = (t == 1) | (t == 2)
    return dict(types=t, pdfs=sim.pdfs()[:, fl], phi=sim.phi(), mass=sim.mass()[t == 1],
                kappa=sim.kappa()[t == 1], counts=sim.counts(), steps=sim.step_count,
                status=sim.status(), trace=sim.trace(n), lost=sim.lost_mass())


@pytest.mark.parametrize("case,prec", [(c, p) for c, (_, ps) in CASES.items() for p in ps])
def test_one_launch_equals_single_steps(fsl, case, prec):
    w = CASES[case][0]()
    n = 60
    got = []
    for parts in ([n], [1] * n, [5, 1, 4, 3, n - 13]):
        sim = fsl.Sim(w["params"], prec)
        sim.init_workload(w)
        sim.set_trace(2)
        for k in parts:
            sim.step(k)
        got.append(_state(sim, n // 2))
        sim.close()
    for other in got[1:]:
        for k, v in got[0].items():
            assert np.array_equal(np.asarray(v), np.asarray(other[k]), equal_nan=True), (case, prec, k)
    if case == "unstable":
        assert got[0]["status"][0] == fsl.ERR_UNSTABLE
