"""Links in the collide kernels where a sphere is free (with fixed spheres
alone the link kernel takes them): a fluid node between three overlapping
spheres, in a lattice of few links per node."""
import numpy as np
import pytest

import oracle
from paper_1808_08921_gb300 import lbmdem
from test_links_fused_gpu import _close, _launches, _run, _three_spheres
from test_parity_gpu import compare_fields, compare_particles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [1, 3])
def test_three_spheres_one_of_them_free(steps):
    w = _three_spheres()
    w.fixed = np.array([1, 1, 0], np.uint8)
    a, b = _run(w, steps, 2), _run(w, steps, 1)
    _close(a, b, 3.0)
    assert _launches(w, steps, 1) - _launches(w, steps, 2) == (steps + 1) // 2
    g, o = lbmdem.Sim.from_workload(w, link_mode=2), oracle.Oracle(w)
    g.step(steps)
    o.step(steps)
    compare_fields(g, o)
    compare_particles(g, o, R=w.R)
    g.close()
    o.close()
