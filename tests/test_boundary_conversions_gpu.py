"""Spheres that cover and uncover nodes beside the inlet and outlet planes while
a call runs many steps: the previous step's inlet / outlet is applied by the
map as it was, next to the blocks that change it.  Against the FP64 oracle
with the bars of test_parity_gpu; also nodes inside two overlapping spheres of
equal and of different radii, whose owner the FP64 rule decides."""
import numpy as np
import pytest

import oracle
import workloads
from paper_1808_08921_gb300 import lbmdem
from test_parity_gpu import compare_fields, compare_particles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("outlet", [workloads.OUTLET_ZERO_GRADIENT, workloads.OUTLET_PRESSURE])
def test_conversions_beside_the_planes(outlet):
    X = np.array([[5.2, 6.0, 6.5], [18.9, 7.2, 6.1], [5.4, 16.0, 17.0], [18.6, 16.3, 17.4]])
    w = workloads.Workload(name="ends", nx=25, ny=24, nz=23, tau=0.8, X=X, R=np.full(4, 3.6), fixed=np.zeros(4, np.uint8),
                           V=np.array([[-0.02, 0, 0], [0.02, 0, 0], [-0.015, 0.004, 0], [0.015, 0, 0.004]]),
                           W=np.zeros((4, 3)), rho_p=20.0, amplitude=2e-3, omega=0.3, dem_substeps=2)
    w.outlet = outlet
    g, o = lbmdem.Sim.from_workload(w, skin=0.9, dem_skin=1.8), oracle.Oracle(w)
    near = 0
    for n in (17, 24):
        s0 = o.fields()[2]
        g.step(n)
        o.step(n)
        compare_fields(g, o)
        compare_particles(g, o, R=w.R)
        s1 = o.fields()[2]
        near += int((s0[1] != s1[1]).sum() + (s0[-2] != s1[-2]).sum())
    assert near > 5 and g.counters()["conversions"] > 20
    g.close()
    o.close()


@pytest.mark.parametrize("R2", [4.0, 3.3])
def test_owner_inside_two_spheres(R2):
    """A mirror plane of lattice nodes between equal spheres: equal distances."""
    X = np.array([[9.0, 8.0, 8.0], [15.0, 8.0, 8.0], [22.3, 8.2, 8.4], [27.1, 8.1, 8.0]])
    w = workloads.Workload(name="lens", nx=36, ny=18, nz=17, tau=0.8, X=X, R=np.array([4.0, R2, 4.0, R2]),
                           fixed=np.zeros(4, np.uint8), V=np.full((4, 3), [0.0, 0.006, 0.004]), W=np.zeros((4, 3)),
                           rho_p=50.0, amplitude=1e-3, omega=0.2, dem_substeps=2)
    g, o = lbmdem.Sim.from_workload(w, skin=0.9, dem_skin=1.8), oracle.Oracle(w)
    for n in (1, 12):
        g.step(n)
        o.step(n)
        compare_fields(g, o)
    g.close()
    o.close()
