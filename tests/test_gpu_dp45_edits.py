"""Dormand-Prince runs whose handle is changed between attempts: the first
stage of the next attempt is taken at the accepted amplitude alpha, whatever
stage the last attempt ended on, and its second stage at the step length then
in use, as the oracle (which keeps nothing from one step to the next) takes
them.

A fast cavity (omega dt of order 1 in a step) with a large amplitude and a weak
coupling makes alpha's own rotation the whole of what is compared: alpha is
FP64 on both sides and the accepted step lengths are the GPU's, so the two
differ by rounding and by the FP32 magnetisation's part in X only.  With
|X| / hbar below omega |alpha| (checked) that part is at most 2^-20 of |alpha|
per radian; 1e-5 |alpha| is allowed for the tens of radians run.  A second
stage at the wrong time or a first one at the wrong amplitude shows at 1e-4 to
1e-2.
"""
import math

import numpy as np
import pytest

from gpu_common import make_pair, require_gpu

pytestmark = pytest.mark.gpu

NX, NY, NZ, D, MS = 12, 10, 2, 1e-8, 1.4e5
WC = (2 * math.pi * 90e9, 2 * math.pi * 70e9)
TOL = 1e-3          # of the controller: steps of a few ps, omega dt of order 1


def _pair(modes=1):
    import oracle
    import paper_2410_00966_gb300 as pkg
    import synthetic
    sim, o = make_pair(NX, NY, NZ, D, MS, 3.65e-12, 0.02)
    m0 = synthetic.tilted_m(NX * NY * NZ, synthetic.derive_seed(95, 1), 0.2)
    sim.set_m(m0)
    o.set_m(m0.astype(np.float64))
    for h in (sim, o):
        h.set_bias((0.05, 0.0, 0.0))
        for k in range(modes):
            h.set_cavity_mode(k, WC[k], 2 * math.pi * 2e7, 2 * math.pi * 5e7)
            h.set_cavity_init_mode(k, 60.0 + 20.0 * k, 25.0)
    sim.set_integrator(pkg.MMCQ_DP45, TOL, pkg.MMCQ_CAVITY_E)
    o.set_integrator(oracle.DP45, TOL, oracle.CAV_E)
    return sim, o


class _Run:
    """Steps the GPU and replays its accepted steps in the oracle."""

    def __init__(self, modes=1):
        self.sim, self.o = _pair(modes)
        self.modes, self.done = modes, 0

    def step(self, n, dt=0.0):
        self.sim.step(n, dt)
        h = self.sim.dt_history()
        self.o.replay(h[self.done:])
        self.done = len(h)

    def both(self, f):
        f(self.sim)
        f(self.o)

    def check(self, label):
        dm = np.abs(self.sim.get_m().astype(np.float64) - self.o.get_m()).max()
        print(f"{label}: {self.done} steps, t = {self.sim.cavity()['t']:.3e}, max|dm| = {dm:.2e}", end="")
        assert self.done >= 8
        errs = []
        for k in range(self.modes):
            c, oc = self.sim.cavity(0, k), self.o.cavity_mode(k)
            a, b = complex(c["re_alpha"], c["im_alpha"]), complex(oc["re_alpha"], oc["im_alpha"])
            assert abs(c["X"]) / 1.05457182e-34 < WC[k] * abs(b)
            errs.append(abs(a - b) / abs(b))
        print("; |d alpha| / |alpha| =", ", ".join(f"{e:.2e}" for e in errs))
        assert dm <= 1e-5
        assert max(errs) <= 1e-5
        self.sim.close()


@pytest.mark.parametrize("edit", ["bias", "m", "ms", "other_mode"])
def test_first_stage_after_an_edit_starts_at_the_accepted_amplitude(edit):
    require_gpu()
    r = _Run(modes=2 if edit == "other_mode" else 1)
    r.step(6, 1e-12)
    for i in range(6):
        if edit == "bias":
            r.both(lambda h: h.set_bias((0.05 + 0.002 * (i % 2), 0.0, 0.0)))
        elif edit == "m":
            m = r.sim.get_m()
            r.sim.set_m(m)
            r.o.set_m(r.sim.get_m().astype(np.float64))
        elif edit == "ms":
            ms = np.full(NX * NY * NZ, MS, np.float32)
            ms[i] = 0.9 * MS
            r.sim.set_ms_map(ms)
            r.o.set_ms(ms.astype(np.float64))
        else:
            r.both(lambda h: h.set_cavity_init_mode(1, 50.0 + i, 10.0))
        r.step(2)
    r.check(edit)


def test_new_step_length_with_a_kept_first_stage():
    """Alternating step lengths given by the caller: the first stage is kept
    (first same as last), the second is at alpha + dt a_21 d alpha/dt for the
    new dt."""
    require_gpu()
    r = _Run()
    r.step(4, 1e-12)
    for i in range(8):
        r.step(1, (8e-13, 2.4e-12)[i % 2])
    r.check("dt")


def test_step_clipped_by_a_new_horizon_with_a_kept_first_stage():
    require_gpu()
    r = _Run()
    r.step(6, 1e-12)
    for i in range(6):
        c = r.sim.cavity()
        r.sim.set_horizon(c["t"] + 0.35 * c["dt"])    # the next attempt is cut to a third
        r.step(1)
        r.sim.set_horizon(0.0)
        r.step(2)
    r.check("horizon")


def test_first_stage_after_a_changed_drive_sees_the_new_drive():
    """The excitation acts in every stage: its change drops the kept first
    stage.  (20 mT over a step of a few ps turns m by some 1e-4 in the first
    stage's share of it.)"""
    require_gpu()
    r = _Run()
    amp = 0.02 / np.abs(r.o.get_brms()).max()
    r.step(6, 1e-12)
    for i in range(6):
        r.both(lambda h: h.set_drive((amp, -0.5 * amp, 0.0)[i % 3], 2 * math.pi * 1e10, r.sim.cavity()["t"]))
        r.step(2)
    r.check("drive")
