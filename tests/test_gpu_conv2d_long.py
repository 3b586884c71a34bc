"""Films of 513 to 1024 rows (y transforms of 2048 points): the demag field
against the oracle, at the edges of that range and with odd sizes.  The bar is
the one of the other field tests: 2e-6 of the largest component."""
import numpy as np
import pytest

from gpu_common import make_pair, require_gpu

pytestmark = pytest.mark.gpu

GRIDS = [(1, 513), (2, 1024), (3, 777), (33, 640), (520, 515), (7, 1023)]


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "x".join(map(str, g)))
def test_field_of_a_long_film_matches_oracle(grid):
    require_gpu()
    import paper_2410_00966_gb300 as pkg
    import synthetic
    nx, ny = grid
    n = nx * ny
    sim, o = make_pair(nx, ny, 1, 4e-9, 8e5, 1.3e-11, 0.01, batch=2)
    ms = synthetic.uniform_ms_map(n, 77, 7e5, 9e5)
    ms[:: 5] = 0.0
    sim.set_ms_map(ms)
    o.set_ms(ms.astype(np.float64))
    sim.set_m(synthetic.random_m(n, 500 + n), inst=0)
    m = synthetic.random_m(n, 900 + n)
    sim.set_m(m, inst=1)
    ref = o.demag(sim.get_m(1).astype(np.float64))
    got = sim.eval_field(pkg.MMCQ_TERM_DEMAG, inst=1)
    assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max()
    # with a plan that shifts the rows of the x passes the field is the same
    plan = sim.tuning()
    sim.set_tuning(dict(plan, x_rows=1))
    assert np.array_equal(sim.eval_field(pkg.MMCQ_TERM_DEMAG, inst=1), got)
    sim.close()
