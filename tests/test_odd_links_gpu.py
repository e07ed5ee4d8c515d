"""The odd steps' links inside the collide kernel (from 65536 stored nodes and
two links per stored node up) against the link kernel every step: FCC packings
with moving spheres and conversions (R 5.5) and with nodes whose solid
neighbours belong to three spheres (R 5.7, 5% of the nodes), block sizes, the
monitored kernels, open and periodic ends; after an odd last step and an
even one.  The bars are those of test_links_fused_gpu (FP32 summation order),
over few steps: contacts amplify it."""
import numpy as np
import pytest

import workloads
from test_links_fused_gpu import _close, _launches, _run

pytestmark = pytest.mark.gpu


def _fcc(R, inlet):
    w = workloads.fcc_column(320, 32, 32, 0.8, 16.0, R, jitter=0.01, seed=4, period=60, substeps=2)
    w.inlet = inlet
    if R < 5.6:  # gaps between the spheres: they move freely
        w.V = np.random.default_rng(3).uniform(-0.01, 0.01, w.X.shape)
    return w


@pytest.mark.parametrize("inlet", [workloads.INLET_PRESSURE, workloads.X_PERIODIC])
@pytest.mark.parametrize("over", [{}, dict(tile=128), dict(tile=256, monitor_every=2)])
@pytest.mark.parametrize("R", [5.5, 5.7])
def test_against_the_link_kernel(R, inlet, over):
    w = _fcc(R, inlet)
    for steps in (2, 13):
        a, b = _run(w, steps, 2, **over), _run(w, steps, 1, **over)
        _close(a, b, R)
    assert a[2]["stored"] >= 65536 and a[2]["links"] >= 2 * a[2]["stored"]
    assert a[2]["conversions"] > 0 or R > 5.6
    assert _launches(w, 4, 1, **over) - _launches(w, 4, 2, **over) == 4
