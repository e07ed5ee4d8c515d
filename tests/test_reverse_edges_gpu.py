"""The reverse kernels at the edges of their ranges: ragged lattices (z lines
that fill no block, partial 32-node words), every outlet, a z segment that
more spheres reach than a block's list holds.  Gradients against central
differences of the FP64 oracle's loss with the bar of test_adjoint_gpu and
test_surrogate_gpu (1e-3)."""
import numpy as np
import pytest

import oracle
import workloads
from paper_1808_08921_gb300 import lbmdem

pytestmark = pytest.mark.gpu

STEPS, EVERY = 60, 20


def _case(outlet, shape, tau=0.8, amp=1e-3):
    nx, ny, nz = shape
    w = workloads.random_small(21, nx=nx, ny=ny, nz=nz, n=5, R=3.2, tau=tau, mobile=False)
    w.outlet, w.amplitude, w.omega, w.probe_x = outlet, amp, 2 * np.pi / 30, 5
    return w


def _oracle_loss(w, target, surrogate):
    o = oracle.Oracle(w)
    o.set_coupling(surrogate)
    o.step(STEPS)
    p = o.probe()[:STEPS] / 3.0
    o.close()
    return float(((p - target) ** 2).sum())


@pytest.mark.parametrize("surrogate", [False, True])
@pytest.mark.parametrize("outlet,shape", [(workloads.OUTLET_PRESSURE, (30, 17, 33)),
                                          (workloads.OUTLET_ZERO_GRADIENT, (30, 13, 40)),
                                          (workloads.OUTLET_WALL, (30, 12, 12))])
def test_gradients_on_ragged_lattices(surrogate, outlet, shape):
    target = np.full(STEPS, 1.0 / 3.0) + np.random.default_rng(1).normal(0.0, 1e-4, STEPS)
    g = lbmdem.Sim.from_workload(_case(outlet, shape))
    out = g.adjoint_psm(STEPS, EVERY, target) if surrogate else g.adjoint(STEPS, EVERY, target)
    g.close()
    h, ha = 1e-4, 1e-6
    fd_tau = (_oracle_loss(_case(outlet, shape, tau=0.8 + h), target, surrogate) -
              _oracle_loss(_case(outlet, shape, tau=0.8 - h), target, surrogate)) / (2 * h)
    fd_amp = (_oracle_loss(_case(outlet, shape, amp=1e-3 + ha), target, surrogate) -
              _oracle_loss(_case(outlet, shape, amp=1e-3 - ha), target, surrogate)) / (2 * ha)
    assert abs(out[1] - fd_tau) <= 1e-3 * abs(fd_tau), (out[1], fd_tau)
    assert abs(out[2] - fd_amp) <= 1e-3 * abs(fd_amp), (out[2], fd_amp)


def test_solid_fraction_where_a_segment_meets_many_spheres():
    """Spheres of radius 0.6 spaced 1.05: over 256 of them within reach of a 256-node z segment."""
    s = np.arange(0, 1, 1.05 / 8)[:-1] * 8
    z = np.arange(0, 255, 1.05)
    X = np.array([[x, y, zz] for x in (5.0, 6.05) for y in s[:6] + 0.5 for zz in z])
    w = workloads.Workload(name="many", nx=12, ny=8, nz=256, tau=0.8, X=X, R=np.full(len(X), 0.6),
                           fixed=np.ones(len(X), np.uint8), amplitude=1e-3, omega=2 * np.pi / 20, probe_x=3,
                           dem_substeps=1)
    near = np.hypot(X[:, 0] - 5.0, X[:, 1] - 3.0) < 1.1
    assert near.sum() > 256
    g = lbmdem.Sim.from_workload(w, skin=0.05, dem_skin=0.2)
    _, tr = g.surrogate_loss(STEPS, np.zeros(STEPS))
    g.close()
    o = oracle.Oracle(w)
    o.set_coupling(True)
    o.step(STEPS)
    ref = o.probe()[:STEPS] / 3.0
    o.close()
    assert np.abs(tr - ref).max() <= 1e-3 * np.abs(ref - ref[0]).max()


@pytest.mark.parametrize("storage", [lbmdem.F32, lbmdem.BF16_DEV])
@pytest.mark.parametrize("R", [3.2, 8.5])
def test_snapshots_of_short_and_odd_runs(storage, R):
    """The reverse sweep's states from the collide kernels: checkpoints every
    2 steps, a run shorter than the interval and an odd last segment give the
    gradient of one segment (FP32 rounding of the same sums); spheres on both
    sides of the radius at which the even steps take their links themselves."""
    n = 4 if R < 5 else 2
    w = workloads.random_small(3, nx=48, ny=24, nz=24, n=n, R=R, tau=0.7, mobile=False)
    assert len(w.R) == n
    w.amplitude, w.omega, w.probe_x = 1e-3, 0.2, 5
    for steps in (7, 24):
        target = np.full(steps, 1.0 / 3.0)
        out = []
        for every in (2, 10, 60):
            g = lbmdem.Sim.from_workload(w, storage=storage, skin=0.1)
            out.append(g.adjoint(steps, every, target))
            g.close()
        for o in out[1:]:
            assert np.array_equal(o[3], out[0][3])
            assert abs(o[1] - out[0][1]) <= 1e-6 * abs(out[0][1])
            assert abs(o[2] - out[0][2]) <= 1e-6 * abs(out[0][2])
