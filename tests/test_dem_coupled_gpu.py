"""More spheres than one cluster of CTAs takes, moving in the fluid, against
the FP64 oracle: the hydrodynamic drive, the lists' life over a re-layout and
the order of a step's kernels where the DEM is a launch per substep.  Touching
spheres, and fast ones apart whose nodes convert.  Bars of test_parity_gpu."""
import numpy as np
import pytest

import oracle
import workloads
from paper_1808_08921_gb300 import lbmdem
from test_parity_gpu import compare_fields, compare_particles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,vel,calls", [(2.85, 0.0, (1, 8, 16)), (2.8, 0.02, (2, 17))])
def test_launches_per_substep_in_the_fluid(R, vel, calls):
    w = workloads.fcc_column(96, 56, 56, 0.8, 8.0, R, jitter=0.003, seed=6, period=40, substeps=4)
    assert len(w.R) == 2352
    if vel:
        w.V = np.where(w.fixed[:, None], 0.0, np.random.default_rng(2).uniform(-vel, vel, w.X.shape))
    g, o = lbmdem.Sim.from_workload(w, skin=0.1), oracle.Oracle(w)
    for n in calls:
        g.step(n)
        o.step(n)
        assert g.status() == 0
        compare_fields(g, o)
        compare_particles(g, o, R=w.R)
    c = g.counters()
    assert c["neighbour_entries"] > 0
    assert not vel or c["conversions"] > 100 and c["relayouts"] > 0
    g.close()
    o.close()
