"""The tuner times what a step launches, whatever its stage buffers hold, and a
plan's rows per x block are run."""
import math
import time

import numpy as np
import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def _sim(nx, ny, nz, batch=1):
    import paper_2410_00966_gb300 as pkg
    import synthetic
    sim = pkg.Sim(nx, ny, nz, 4e-9, 4e-9, 4e-9, 8e5, 1.3e-11, 0.01, batch=batch)
    sim.set_m(synthetic.tilted_m(nx * ny * nz, synthetic.derive_seed(96, nx), 0.2))
    sim.set_bias((0.05, 0.0, 0.0))
    sim.set_cavity(2 * math.pi * 5e9, 2 * math.pi * 1e7, 2 * math.pi * 2e8)
    sim.set_cavity_init(2.0, 0.0)
    return sim


@pytest.mark.parametrize("grid", [(40, 40, 1), (72, 40, 6)], ids=lambda g: "x".join(map(str, g)))
def test_the_timed_stage_takes_as_long_as_a_stage_of_a_step(grid):
    """The plan's time is that of a stage as steps launch it: its kernels in a
    row, each placed as the one before ends, and the scalar work beside the x
    forward.  25 % covers the start of a short chain (some 4 us in 80) and the
    difference between a middle stage and the mean of four."""
    require_gpu()
    sim = _sim(*grid)
    sim.step(4, 5e-14)
    plan = sim.autotune(reps=9)
    sim.step(100, 5e-14)
    sim.sync()
    best = math.inf
    for _ in range(5):
        t = time.perf_counter()
        sim.step(200, 5e-14)
        sim.sync()
        best = min(best, (time.perf_counter() - t) / 800 * 1e3)
    print(f"stage of {grid}: tuner {plan['eval_ms'] * 1e3:.2f} us (rules {plan['rule_ms'] * 1e3:.2f}), steps {best * 1e3:.2f} us")
    sim.close()
    assert 0.75 * best <= plan["eval_ms"] <= 1.25 * best


@pytest.mark.parametrize("kind", [0, 1], ids=["rk4", "dp45"])
def test_tuning_a_new_handle_leaves_no_error(kind):
    """The timed stage reads stage buffers that no step has written yet: what
    happens to be in that memory (here NaN) is no error of the run."""
    require_gpu()
    import torch
    import paper_2410_00966_gb300 as pkg
    nx, ny, nz = 44, 36, 3
    _sim(nx, ny, nz).close()                      # (the library is loaded)
    torch.cuda.empty_cache()
    sizes = [16 * nx * ny * nz] * 16 + [1 << 21] * 4 + [1 << 16] * 40
    junk = [torch.full((s // 4,), float("nan"), device="cuda") for s in sizes]
    torch.cuda.synchronize()
    del junk                                      # back to the allocator that the handle takes its buffers from
    sim = _sim(nx, ny, nz)
    sim.set_integrator(kind, 1e-6, pkg.MMCQ_CAVITY_E)
    sim.autotune(reps=2)
    sim.step(3, 1e-14)
    sim.sync()
    assert np.isfinite(sim.get_m()).all()
    sim.close()


def test_rows_of_a_plan_are_run_as_given():
    """Fewer rows per x block than the largest count are a choice of the
    caller's, not a bound: on a 32x32 film the rule runs one row per block, and
    a plan of 31 runs two blocks, whose load, transform and store loops go
    through their rows one after the other (x passes of 32 rows per block take
    three times as long as of one, which is more than 15 % of the stage).  The
    field is the same."""
    require_gpu()
    import paper_2410_00966_gb300 as pkg
    sim = _sim(32, 32, 1)
    rule = sim.tuning()
    assert rule["x_rows"] == 32
    t, f = {}, {}
    for rows in (32, 31):
        sim.set_tuning(dict(rule, x_rows=rows))
        f[rows] = sim.eval_field(pkg.MMCQ_TERM_DEMAG)
    for rows in (32, 31):
        sim.set_tuning(dict(rule, x_rows=rows))
        assert sim.tuning()["x_rows"] == rows
        t[rows] = math.inf
        for _ in range(5):
            t0 = time.perf_counter()
            sim.step(200, 5e-14)
            sim.sync()
            t[rows] = min(t[rows], time.perf_counter() - t0)
    print(f"rows: stage {t[32] / 800 * 1e6:.2f} us under the rule, {t[31] / 800 * 1e6:.2f} us with 31 rows per block")
    sim.close()
    assert np.array_equal(f[31], f[32])
    assert t[31] > 1.15 * t[32]
