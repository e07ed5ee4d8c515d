"""What lbm_dem_adjoint leaves behind: the context at t0 + steps, as a plain
run of the same steps does, whatever the segments; even and odd counts, a last
segment of one step.  The fluid of a fixed packing is a deterministic function
of its state, so the fields are equal bit for bit; plane means and probe, force
and torque and the gradient to the order of their FP64 sums."""
import numpy as np
import pytest

import workloads
from paper_1808_08921_gb300 import lbmdem

pytestmark = pytest.mark.gpu


def _sim(storage):
    w = workloads.random_small(9, nx=33, ny=13, nz=35, n=5, R=2.7, mobile=False)
    w.amplitude, w.omega, w.probe_x = 3e-3, 0.3, 4
    return lbmdem.Sim.from_workload(w, storage=storage)


def _same(a, b):
    assert all(np.array_equal(x, y) for x, y in zip(a.fields(), b.fields()))
    for x, y in zip(a.plane_means() + (a.probe(),), b.plane_means() + (b.probe(),)):
        assert x.shape == y.shape and np.abs(x - y).max() <= 1e-13
    p, q = a.particles(), b.particles()
    assert np.abs(q["Fh"]).max() > 0 or a.counters()["t"] < 8  # the wave has to reach a sphere first
    for k in ("Fh", "Th"):
        assert np.abs(p[k] - q[k]).max() <= 1e-9 * np.abs(q[k]).max()
    assert a.counters()["t"] == b.counters()["t"]


@pytest.mark.parametrize("storage", [lbmdem.F32, lbmdem.BF16_DEV])
@pytest.mark.parametrize("before,steps,every", [(0, 24, 24), (0, 24, 6), (2, 25, 8), (18, 17, 16), (0, 3, 2)])
def test_context_after_the_gradient(before, steps, every, storage):
    target = np.full(steps, 1 / 3)
    a, b = _sim(storage), _sim(storage)
    for s in (a, b):
        s.step(before)
    a.adjoint(steps, every, target)
    b.step(steps)
    _same(a, b)
    for s in (a, b):  # an odd step count reached, then an even one
        s.step(1)
    _same(a, b)
    n = 17 - (before + steps) % 2
    for s in (a, b):
        s.step(n)
    _same(a, b)
    assert a.counters()["t"] % 2 == 0
    # and another gradient from there
    la, lb = a.adjoint(8, 4, np.full(8, 1 / 3)), b.adjoint(8, 4, np.full(8, 1 / 3))
    assert np.abs(la[3] - lb[3]).max() <= 1e-13
    for x, y in zip(la[:3], lb[:3]):
        assert abs(x - y) <= 1e-8 * abs(y)
    _same(a, b)
    a.close()
    b.close()
