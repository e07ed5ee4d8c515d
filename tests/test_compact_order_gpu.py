"""The compact order at the edges of its 32-node words: z lines of one node,
one short of, one, and one past a whole number of words, and their wrap;
single lines in y.  Against the FP64 oracle with the bars of
test_parity_gpu.  A packing of fixed spheres stores fluid nodes only, one
with a free sphere some solid ones too."""
import numpy as np
import pytest

import oracle
import workloads
from paper_1808_08921_gb300 import lbmdem
from test_parity_gpu import compare_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inlet", [workloads.INLET_PRESSURE, workloads.X_PERIODIC])
@pytest.mark.parametrize("ny,nz", [(1, 1), (1, 33), (3, 31), (2, 64), (12, 32), (12, 65), (33, 12)])
@pytest.mark.parametrize("mobile", [False, True])
def test_words(ny, nz, inlet, mobile):
    room = ny >= 12 and nz >= 12
    if not room and mobile or not mobile and inlet == workloads.X_PERIODIC:
        pytest.skip("no sphere, or nothing that moves: a fluid at rest")
    w = workloads.random_small(2, nx=21, ny=max(ny, 12), nz=max(nz, 12), n=4, R=2.4, mobile=mobile, vel=0.03)
    w.ny, w.nz, w.inlet, w.amplitude, w.omega = ny, nz, inlet, 2e-3, 0.3
    w.body_force = (1e-4, 2e-5, 3e-5) if mobile else (0.0, 0.0, 0.0)
    if not room:
        w.X, w.R, w.fixed, w.V, w.W = np.zeros((0, 3)), np.zeros(0), np.zeros(0, np.uint8), None, None
    g, o = lbmdem.Sim.from_workload(w), oracle.Oracle(w)
    for n in (1, 2, 16):
        g.step(n)
        o.step(n)
        compare_fields(g, o)
    c = g.counters()
    assert (c["stored"] > c["fluid"]) if mobile else (c["stored"] == c["fluid"])
    g.close()
    o.close()
