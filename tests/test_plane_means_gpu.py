"""Plane means against the means of the read-out fields, over ragged lattices
and both parities, to the FP32 rounding of a node's 19-term sums."""
import numpy as np
import pytest

import workloads
from paper_1808_08921_gb300 import lbmdem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(19, 13, 37), (64, 16, 16), (5, 33, 70)])
@pytest.mark.parametrize("steps", [21, 40])
def test_plane_means_are_the_fields_means(shape, steps):
    nx, ny, nz = shape
    w = workloads.random_small(4, nx=nx, ny=ny, nz=nz, n=6 if nx > 12 else 0, R=2.6, vel=0.02)
    if nx <= 12:  # no room for spheres: a pure fluid
        w.X, w.R, w.fixed, w.V, w.W = np.zeros((0, 3)), np.zeros(0), np.zeros(0, np.uint8), None, None
    w.amplitude, w.omega = 2e-3, 0.2
    g = lbmdem.Sim.from_workload(w)
    g.step(steps)
    rho, u, solid = g.fields()
    mean_rho, mean_jx = g.plane_means()
    g.close()
    fl = solid == 0
    cnt = fl.sum((1, 2))
    rho_p = np.where(fl, rho, 0.0).sum((1, 2)) / cnt
    jx_p = np.where(fl, rho * u[0], 0.0).sum((1, 2)) / cnt
    # a node's FP32 sum of 19 deviations: 19 roundings of at most the largest
    # deviation, itself below |rho - 1| + 3 |u|
    tol = 19 * 2.0 ** -24 * (np.abs(rho[fl] - 1.0).max() + 3 * np.abs(u).max())
    assert np.abs(mean_rho - rho_p).max() <= tol
    assert np.abs(mean_jx - jx_p).max() <= tol
