"""The DEM's launches at the edges of their ranges, spheres alone, against the
FP64 oracle: one CTA, one cluster of CTAs (full and with one sphere more than
a CTA's share), one launch per substep; lists longer than the entries held in
registers (a wide skin); fixed spheres among them.  Bars of test_parity_gpu
for centres, velocities of their largest."""
import numpy as np
import pytest

import oracle
import workloads
from paper_1808_08921_gb300 import lbmdem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,skin", [(1, 0.5), (3, 0.5), (64, 0.5), (65, 0.5), (64, 4.0), (129, 4.0), (1024, 0.5),
                                    (1025, 2.0), (2047, 0.5), (2048, 0.5), (2049, 0.5), (2500, 2.0)])
def test_spheres_alone(n, skin):
    rng = np.random.default_rng(n)
    R, side = 3.0, max(4, int(np.ceil(n ** (1 / 3))))
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    X = 4.0 + 6.0 * g + rng.uniform(-0.02, 0.02, (n, 3))  # touching neighbours: gaps and overlaps of 0.04
    L = 6 * side + 2
    fixed = (rng.uniform(size=n) < 0.1).astype(np.uint8)
    fixed[0] = 0
    V = np.where(fixed[:, None], 0.0, rng.uniform(-1e-3, 1e-3, (n, 3)))
    W = np.where(fixed[:, None], 0.0, rng.uniform(-1e-3, 1e-3, (n, 3)))
    w = workloads.Workload(name="dry", nx=L, ny=L, nz=L, tau=0.8, X=X, R=np.full(n, R), fixed=fixed, V=V, W=W,
                           dem_substeps=5, body_force=(1e-5, 0.0, -2e-5))
    s = lbmdem.Sim(lbmdem.params_from_workload(w, lbm_on=0, dem_skin=skin))
    s.set_packing(w.X, w.R, w.V, w.W, w.fixed)
    o = oracle.Oracle(w, lbm_on=False)
    for steps in (1, 9):
        s.step(steps)
        o.step(steps)
        a, b = s.particles(), o.particles()
        assert s.status() == 0
        assert np.abs(a["X"] - b["X"]).max() <= 1e-6
        for k, scale in (("V", np.abs(b["V"]).max()), ("W", max(np.abs(b["W"]).max(), np.abs(b["V"]).max() / R))):
            assert np.abs(a[k] - b[k]).max() <= 1e-3 * scale, k
        assert np.abs(a["q"] - b["q"]).max() <= 1e-5
    if n > 1:
        assert s.counters()["neighbour_entries"] > 0
    s.close()
    o.close()
