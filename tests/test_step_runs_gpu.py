"""The same steps taken in one call, in uneven calls and one at a time: inside
a call a step leaves its inlet / outlet to the next step's first kernel, at
its end the state is complete.  Fixed spheres: the fluid is a deterministic
function of its state, so the results are equal bit for bit; free spheres:
their FP64 sums are formed in any order, so equal to FP32 rounding."""
import numpy as np
import pytest

import workloads
from paper_1808_08921_gb300 import lbmdem

pytestmark = pytest.mark.gpu


def _run(w, calls, **over):
    s = lbmdem.Sim.from_workload(w, **over)
    for n in calls:
        s.step(n)
    assert s.status() == 0
    out = s.fields() + (s.probe(), s.monitors(), s.particles()["X"])
    c = s.counters()
    s.close()
    return out, c


@pytest.mark.parametrize("storage", [lbmdem.F32, lbmdem.F16_DEV])
@pytest.mark.parametrize("inlet,outlet", [(workloads.INLET_PRESSURE, workloads.OUTLET_ZERO_GRADIENT),
                                          (workloads.INLET_PRESSURE, workloads.OUTLET_PRESSURE),
                                          (workloads.X_WALL, workloads.OUTLET_PRESSURE),
                                          (workloads.X_PERIODIC, workloads.OUTLET_WALL)])
def test_runs_do_not_depend_on_the_calls(storage, inlet, outlet):
    w = workloads.random_small(9, nx=33, ny=13, nz=35, n=5, R=2.7, mobile=False)
    w.inlet, w.outlet, w.amplitude, w.omega, w.probe_x = inlet, outlet, 3e-3, 0.3, 4
    if inlet == workloads.X_PERIODIC:  # no source: a moving sphere drives the fluid
        w.fixed, w.body_force = np.zeros(5, np.uint8), (0.01, 0.0, 0.0)
    a, ca = _run(w, [37], storage=storage)
    for calls in ([1] * 37, [2, 16, 3, 15, 1], [5, 32]):
        b, cb = _run(w, calls, storage=storage)
        assert np.array_equal(a[2], b[2]) and ca["conversions"] == cb["conversions"]
        for x, y in zip(a, b):
            if inlet == workloads.X_PERIODIC:
                assert np.abs(np.asarray(x, float) - y).max() <= 1e-6 * np.abs(y).max()
            else:
                assert np.array_equal(x, y)


def test_conversions_in_runs_and_single_steps():
    """Fast spheres: nodes covered and uncovered before even and odd steps."""
    w = workloads.random_small(5, nx=40, ny=20, nz=20, n=8, R=3.5, vel=0.03)
    a, ca = _run(w, [41], skin=1.0, dem_skin=2.0)
    b, cb = _run(w, [1] * 41, skin=1.0, dem_skin=2.0)
    assert ca["conversions"] == cb["conversions"] > 100
    assert np.array_equal(a[2], b[2])
    assert np.abs(a[1] - b[1]).max() <= 2e-6 * np.abs(b[1]).max()
    assert np.abs(a[5] - b[5]).max() <= 1e-9
