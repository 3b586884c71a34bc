"""A group keeps nothing of a handle that the handle has changed since the
capture: after a coupling map is given to a mode that had none (the map's
buffer is allocated then), grouped steps equal the same handles stepped one by
one bit for bit, for call lengths with and without a remainder."""
import numpy as np
import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

SHAPES = [(24, 20, 1), (16, 8, 3)]


def _handles(pkg, synthetic, kind):
    out = []
    for k, (nx, ny, nz) in enumerate(SHAPES):
        sim = pkg.Sim(nx, ny, nz, 4e-9, 4e-9, 4e-9, 8e5, 1.3e-11, 0.01)
        sim.set_m(synthetic.tilted_m(nx * ny * nz, synthetic.derive_seed(52, k), 0.05))
        sim.set_bias((0.05, 0.0, 0.0))
        sim.set_cavity(2 * np.pi * 5e9, 2 * np.pi * 1e7, 2 * np.pi * 5e8)
        sim.set_cavity_init(20.0, 5.0)
        sim.set_integrator(kind, 1e-6, pkg.MMCQ_CAVITY_E)
        out.append(sim)
    return out


@pytest.mark.parametrize("n", [8, 11], ids=["whole", "remainder"])
@pytest.mark.parametrize("kind", [0, 1], ids=["rk4", "dp45"])
def test_map_given_after_the_capture(kind, n):
    require_gpu()
    import paper_2410_00966_gb300 as pkg
    import synthetic
    direct, grouped = _handles(pkg, synthetic, kind), _handles(pkg, synthetic, kind)
    g = pkg.Group(grouped, chunk=4)
    dt = 5e-14
    for s in direct:
        s.step(n, dt)
    g.step(n, dt)
    for sims in (direct, grouped):
        nx, ny, nz = SHAPES[1]
        prof = np.random.default_rng(5).normal(size=(nx * ny * nz, 3)).astype(np.float32)
        sims[1].set_cavity(2 * np.pi * 5e9, 2 * np.pi * 1e7, 2 * np.pi * 5e8, profile=prof)
    for s in direct:
        s.step(n, dt)
    g.step(n, dt)
    assert g.replays() == 2 * (n // 4)
    for a, b in zip(direct, grouped):
        assert np.array_equal(a.get_m(), b.get_m())
        ca, cb = a.cavity(), b.cavity()
        for key in ("t", "re_alpha", "im_alpha", "dt", "accepted", "rejected"):
            assert ca[key] == cb[key], key
    g.close()
    for s in direct + grouped:
        s.close()
