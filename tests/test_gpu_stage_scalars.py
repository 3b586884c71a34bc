"""The scalar work of a stage (coupling sums, cavity amplitudes, history) is
done by the next stage's x forward within a call and by the stage itself at
its end: a call of n steps gives bit for bit what n calls of one step give."""
import math

import numpy as np
import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

# one row; ragged rows of one and of several per block; three tiles of kx; 3-D
GRIDS = [(1, 1, 1), (9, 1, 3), (33, 20, 1), (100, 7, 2), (16, 400, 1), (260, 5, 9)]


def _run(grid, kind, cavity, modes, calls):
    import paper_2410_00966_gb300 as pkg
    import synthetic
    nx, ny, nz = grid
    n = nx * ny * nz
    sim = pkg.Sim(nx, ny, nz, 4e-9, 4e-9, 4e-9, 8e5, 1.3e-11, 0.01, batch=2)
    for b in range(2):
        sim.set_m(synthetic.tilted_m(n, synthetic.derive_seed(81, b), 0.3), inst=b)
        sim.set_bias((0.05 + 0.01 * b, 0.0, 0.0), inst=b)
        for k in range(modes):
            sim.set_cavity_mode(k, 2 * math.pi * (5e9 + 1e9 * k), 2 * math.pi * 1e7, 2 * math.pi * 2e8, inst=b)
    sim.set_cavity_init(1.0, 0.5)
    sim.set_drive(1e3, 2 * math.pi * 2e10, 1e-12)
    sim.set_recording(1)
    sim.set_integrator(kind, 1e-6, cavity)
    first = True
    for c in calls:
        sim.step(c, 5e-14 if first or kind == pkg.MMCQ_RK4 else 0.0)
        first = False
    out = [sim.get_m(b) for b in range(2)] + [sim.mavg_history(b) for b in range(2)]
    out += [np.array([list(sim.cavity(b, k).values()) for b in range(2) for k in range(modes)])]
    sim.close()
    return out


@pytest.mark.parametrize("modes", [1, 3])
@pytest.mark.parametrize("cavity", ["E", "P"])
@pytest.mark.parametrize("kind", ["rk4", "dp45"])
@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "x".join(map(str, g)))
def test_steps_in_one_call_equal_single_steps(grid, kind, cavity, modes):
    require_gpu()
    import paper_2410_00966_gb300 as pkg
    k = pkg.MMCQ_RK4 if kind == "rk4" else pkg.MMCQ_DP45
    c = pkg.MMCQ_CAVITY_E if cavity == "E" else pkg.MMCQ_CAVITY_P
    a = _run(grid, k, c, modes, [5])
    b = _run(grid, k, c, modes, [1] * 5)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
