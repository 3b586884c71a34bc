"""The scalar work of a Dormand-Prince stage, which the next stage's x forward
does, against the oracle: amplitudes and accumulators of one, two and three
modes, the excitation's time, the recorded averages and the times of the
samples, on grids whose x blocks hold one row, several and ragged ones.  (A call
of five attempts enqueues the same launches as five calls of one, so their
equality says nothing here.)

The oracle replays the accepted step lengths.  m to 1e-5; amplitudes and
accumulators, FP64 on both sides but for X of the FP32 m (1e-6 of sum|terms| at
the most, which is |X| for nearly uniform m), to 1e-5 of their size; the
recorded averages, of a few rounded steps' m, to 1e-6.
"""
import math

import numpy as np
import pytest

from gpu_common import make_pair, require_gpu

pytestmark = pytest.mark.gpu

GRIDS = [(9, 1, 3), (33, 20, 1), (100, 7, 2), (260, 5, 9)]


@pytest.mark.parametrize("modes", [1, 2, 3])
@pytest.mark.parametrize("cavity", [0, 1], ids=["E", "P"])
@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "x".join(map(str, g)))
def test_attempts_match_the_oracle(grid, cavity, modes):
    require_gpu()
    import synthetic
    nx, ny, nz = grid
    n = nx * ny * nz
    sim, o = make_pair(nx, ny, nz, 4e-9, 8e5, 1.3e-11, 0.01)
    m0 = synthetic.tilted_m(n, synthetic.derive_seed(83, modes), 0.2)
    sim.set_m(m0)
    o.set_m(m0.astype(np.float64))
    for h in (sim, o):
        h.set_bias((0.05, 0.0, 0.01))
        for k in range(modes):
            h.set_cavity_mode(k, 2 * math.pi * (3e10 + 1e10 * k), 2 * math.pi * 1e8, 2 * math.pi * 2e8)
            h.set_cavity_init_mode(k, 5.0 - k, 0.5)
        h.set_drive(1e3, 2 * math.pi * 2e11, 2e-13)
        h.set_integrator(1, 1e-5, cavity)
    sim.set_recording(1)
    o.set_recording(True)
    for c in (7, 1, 4):
        sim.step(c, 1e-13 if c == 7 else 0.0)
    hist = sim.dt_history()
    assert len(hist) >= 6
    o.replay(hist)
    assert np.abs(sim.get_m().astype(np.float64) - o.get_m()).max() <= 1e-5
    for k in range(modes):
        c, oc = sim.cavity(0, k), o.cavity_mode(k)
        pair = ("re_alpha", "im_alpha") if cavity == 0 else ("S", "C")
        size = math.hypot(oc[pair[0]], oc[pair[1]])
        err = max(abs(c[q] - oc[q]) for q in pair) / size
        print(f"{grid} mode {k} of {modes}, {'EP'[cavity]}: {len(hist)} steps, error {err:.1e}")
        assert err <= 1e-5
        assert c["t"] == pytest.approx(hist.sum(), rel=1e-12)
    g, r = sim.mavg_history(), o.mavg_history()
    assert g.shape == r.shape == (len(hist), 4)
    assert np.abs(g[:, 0] - r[:, 0]).max() <= 1e-12 * r[-1, 0]
    assert np.abs(g[:, 1:] - r[:, 1:]).max() <= 1e-6
    sim.close()
