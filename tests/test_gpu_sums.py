"""The sums over cells of a stage keep what their FP32 terms hold.

Each thread, block and instance adds the terms of the coupling sum X and of the
recorded average of m in three floats with the error of every addition carried
on, and the result is read out in FP64.  Here the terms are formed on the host
in the kernel's arithmetic (with a map along y the term of a cell is Ms
fl(m_y B_y): one FP32 rounding, then an exact product) and summed exactly
(math.fsum).

Bound: the FP64 operations between the sum and the read-out (a product with
V_c, one with exp, cos and dt each, and back: 8 roundings of 2^-53 of |X|),
1e-15 |X|; and what the third float drops, below 2^-68 of the sum of |terms|
for each of some 2^12 additions per thread and 2^12 merges, 1e-16 of the sum of
|terms|.  Signs alternate, so that |X| is far below that sum; an FP32 sum is
off by 1e-8 of it, one of products rounded to FP32 by 1e-10, an addition whose
term is rounded in one place and not in the other by 1e-11.
"""
import math

import numpy as np
import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

# small blocks of few rows; ragged rows; the compile-time shape; pipelined rows
GRIDS = [(40, 24, 6), (100, 7, 2), (300, 200, 1), (256, 64, 16), (1024, 40, 4)]


def _run(grid, modes):
    import paper_2410_00966_gb300 as pkg
    import synthetic
    nx, ny, nz = grid
    n = nx * ny * nz
    d = 4e-9
    rng = np.random.default_rng(n + modes)
    sim = pkg.Sim(nx, ny, nz, d, d, d, 8e5, 1.3e-11, 0.01)
    ms = (rng.uniform(0.7e6, 0.9e6, n) * (rng.uniform(size=n) > 0.1)).astype(np.float32)
    sim.set_ms_map(ms)
    sim.set_m(synthetic.random_m(n, synthetic.derive_seed(99, modes)))
    sim.set_bias((0.02, 0.01, 0.0))
    wc, kappa, dt = 2 * math.pi * 6e9, 2 * math.pi * 1e7, 1e-13
    maps = []
    for k in range(modes):
        b = np.zeros((n, 3), np.float32)
        b[:, 1] = rng.normal(size=n).astype(np.float32) * np.float32(1e-6)
        maps.append(b[:, 1].copy())
        sim.set_cavity_mode(k, wc, kappa, profile=b, profile_is_brms=True)
    sim.set_recording(1)
    sim.set_integrator(pkg.MMCQ_RK4, 0.0, pkg.MMCQ_CAVITY_P)
    sim.step(1, dt)
    m = sim.get_m()
    out = []
    for k in range(modes):
        c = sim.cavity(0, k)
        t = c["t_cav"]
        out.append(c["C"] / (math.exp(kappa * t) * math.cos(wc * t) * dt))
    avg = sim.mavg_history()
    sim.close()
    return ms, m, maps, out, avg, d ** 3


@pytest.mark.parametrize("modes", [1, 2, 3])
@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: "x".join(map(str, g)))
def test_sums_are_those_of_their_terms(grid, modes):
    require_gpu()
    ms, m, maps, got, avg, vc = _run(grid, modes)
    for k in range(modes):
        assert m.dtype == ms.dtype == maps[k].dtype == np.float32
        terms = ms.astype(np.float64) * (m[:, 1] * maps[k]).astype(np.float64)     # 48 bits: exact
        x, scale = math.fsum(terms) * vc, math.fsum(np.abs(terms)) * vc
        print(f"{grid} mode {k} of {modes}: |X| / sum|terms| = {abs(x) / scale:.1e}, "
              f"error {abs(got[k] - x) / scale:.1e} of sum|terms|")
        assert abs(got[k] - x) <= 1e-15 * abs(x) + 1e-16 * scale
    on = ms > 0
    nm = int(on.sum())
    for c in range(3):
        v = m[on, c].astype(np.float64)
        mean, scale = math.fsum(v) / nm, math.fsum(np.abs(v)) / nm
        print(f"{grid} <m_{'xyz'[c]}>: error {abs(avg[0, 1 + c] - mean) / scale:.1e} of <|m|>")
        assert abs(avg[0, 1 + c] - mean) <= 1e-15 * abs(mean) + 1e-16 * scale
