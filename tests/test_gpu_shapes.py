"""Kernel shapes that need a grid of some size, against the oracle.

* The compile-time x passes of rows of 256 and 512 cells (whole blocks of four
  rows) run where four rows per block leave two blocks on every SM: 913 rows of
  the batch and more on 152 SMs.
* The y passes of 512 and 1024 points of a 3-D grid, one component per block.
* The x inverse with two cavity modes compiled in, plain and recording.

Tolerances are those of the field tests (2e-6 of the largest field: some 20
times log2(P) 2^-24) and of the trajectory tests (1e-5 in m, 1e-4 in alpha).
"""
import math

import numpy as np
import pytest

from gpu_common import make_pair, require_gpu

pytestmark = pytest.mark.gpu

FIXED = [(256, 64, 16), (512, 64, 16)]
LONG_Y = [(16, 200, 3), (40, 257, 2), (16, 512, 3)]


def _alpha(c):
    return complex(c["re_alpha"], c["im_alpha"])


@pytest.mark.parametrize("grid", FIXED + LONG_Y, ids=lambda g: "x".join(map(str, g)))
def test_field(grid):
    require_gpu()
    import paper_2410_00966_gb300 as pkg
    import synthetic
    nx, ny, nz = grid
    n = nx * ny * nz
    sim, o = make_pair(nx, ny, nz, 4e-9, 8e5, 1.3e-11, 0.01)
    ms = synthetic.uniform_ms_map(n, 78, 7e5, 9e5)
    ms[:: 7] = 0.0
    sim.set_ms_map(ms)
    o.set_ms(ms.astype(np.float64))
    sim.set_m(synthetic.random_m(n, 600 + n))
    m = sim.get_m().astype(np.float64)
    for term, ref in ((pkg.MMCQ_TERM_DEMAG, o.demag(m)), (pkg.MMCQ_TERM_EXCHANGE, o.exchange(m))):
        got = sim.eval_field(term)
        assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max()
    # one row per block (no compile-time shape): the same transforms, the same bits
    got = sim.eval_field(pkg.MMCQ_TERM_DEMAG)
    sim.set_tuning(dict(sim.tuning(), x_rows=1))
    assert np.array_equal(sim.eval_field(pkg.MMCQ_TERM_DEMAG), got)
    sim.close()


@pytest.mark.parametrize("kind", [0, 1], ids=["rk4", "dp45"])
@pytest.mark.parametrize("grid", FIXED, ids=lambda g: "x".join(map(str, g)))
def test_steps_of_the_fixed_x_shapes(grid, kind):
    require_gpu()
    import synthetic
    nx, ny, nz = grid
    n = nx * ny * nz
    sim, o = make_pair(nx, ny, nz, 5e-9, 1.4e5, 3.65e-12, 1e-3, Ku=1e3)
    m0 = synthetic.tilted_m(n, synthetic.derive_seed(97, nx), 0.2)
    prof = synthetic.lorentzian_profile(nx, ny, nz, 5e-9, 300e-9, direction=(0.0, 1.0, 0.0))
    sim.set_m(m0)
    o.set_m(m0.astype(np.float64))
    for h, p in ((sim, prof), (o, prof.astype(np.float64))):
        h.set_bias((0.1, 0.0, 0.0))
        h.set_cavity(2 * math.pi * 5e9, 2 * math.pi * 1e7, 2 * math.pi * 2e8, profile=p)
        h.set_cavity_init(2.0, 0.5)
        h.set_integrator(kind, 1e-6, 0)
    if kind == 0:
        sim.step(3, 2e-13)
        o.step(3, 2e-13)
    else:
        sim.step(4, 1e-13)
        hist = sim.dt_history()
        assert len(hist) >= 2
        o.replay(hist)
    dm = np.abs(sim.get_m().astype(np.float64) - o.get_m()).max()
    a, b = _alpha(sim.cavity()), _alpha(o.cavity())
    print(f"{grid} kind {kind}: max|dm| = {dm:.2e}, |d alpha| / |alpha| = {abs(a - b) / abs(b):.2e}")
    assert dm <= 1e-5
    assert abs(a - b) <= 1e-4 * abs(b)
    sim.close()


@pytest.mark.parametrize("cavity", [0, 1], ids=["E", "P"])
@pytest.mark.parametrize("kind", [0, 1], ids=["rk4", "dp45"])
@pytest.mark.parametrize("record", [0, 1], ids=["plain", "recording"])
def test_two_modes(kind, cavity, record):
    require_gpu()
    import synthetic
    nx, ny, nz = 33, 20, 3
    n = nx * ny * nz
    sim, o = make_pair(nx, ny, nz, 4e-9, 8e5, 1.3e-11, 0.01)
    m0 = synthetic.tilted_m(n, synthetic.derive_seed(98, kind), 0.1)
    prof = np.random.default_rng(98).normal(size=(n, 3)).astype(np.float32)
    sim.set_m(m0)
    o.set_m(m0.astype(np.float64))
    for h, p in ((sim, prof), (o, prof.astype(np.float64))):
        h.set_bias((0.05, 0.0, 0.0))
        h.set_cavity_mode(0, 2 * math.pi * 6e9, 2 * math.pi * 2e7, 2 * math.pi * 3e8)
        h.set_cavity_mode(1, 2 * math.pi * 7.5e9, 2 * math.pi * 5e7, 2 * math.pi * 2e8, profile=p)
        for k in range(2):
            h.set_cavity_init_mode(k, 0.3 * (k + 1), -0.1)
        h.set_integrator(kind, 1e-6, cavity)
    if record:
        sim.set_recording(1)
        o.set_recording(True)
    sim.step(40, 1e-13)
    if kind == 0:
        o.step(40, 1e-13)
    else:
        o.replay(sim.dt_history())
    assert np.abs(sim.get_m().astype(np.float64) - o.get_m()).max() <= 1e-5
    for k in range(2):
        a, b = _alpha(sim.cavity(0, k)), _alpha(o.cavity_mode(k))
        if cavity == 0:
            assert abs(a - b) <= 1e-4 * abs(b)
        else:
            c, oc = sim.cavity(0, k), o.cavity_mode(k)
            for q in ("S", "C"):
                assert abs(c[q] - oc[q]) <= 1e-4 * math.hypot(oc["S"], oc["C"])
    if record:
        g, r = sim.mavg_history(), o.mavg_history()
        assert g.shape == r.shape and len(g) > 10
        assert np.abs(g[:, 0] - r[:, 0]).max() <= 1e-12 * r[-1, 0]
        assert np.abs(g[:, 1:] - r[:, 1:]).max() <= 1e-5
    sim.close()
