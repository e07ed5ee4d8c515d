"""Links in the collide kernels where a sphere is free (with fixed spheres
alone the link kernel takes them): a fluid node between three overlapping
spheres, in a lattice of few links per node; and which lattices count as ones
of few links."""
import numpy as np
import pytest

import oracle
import workloads
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


@pytest.mark.parametrize("a,R,cx,odd", [(13, 2.5, 10, False), (12, 2.5, 12, False), (16, 3.5, 6, True)])
def test_two_links_per_stored_node(a, R, cx, odd):
    """Small spheres' link records are padded to three and four times their
    number; the odd steps take their links by the number without padding."""
    w = workloads.fcc_column(a * cx, 2 * a, 2 * a, 0.8, float(a), R, jitter=0.01, seed=4, period=60, substeps=2)
    c = _run(w, 4, 2)[2]
    assert c["stored"] >= 65536 and (c["links"] >= 2 * c["stored"]) == odd
    assert 0.75 < c["links"] / (2 * c["stored"]) < 1.25
    assert _launches(w, 4, 1) - _launches(w, 4, 2) == (4 if odd else 2)
