"""A dense FCC packing of fixed spheres of radius 8 lu and more, FP32: only the
last step of a call takes its links there, and neither the calls a run is split
into, nor the steps of a graph, nor a gradient's segments show in the fluid,
bit for bit; in the probe, the sphere forces and the gradient not beyond the
order of their FP64 sums."""
import numpy as np
import pytest

import workloads
from paper_1808_08921_gb300 import lbmdem

pytestmark = pytest.mark.gpu


def _sim(**over):
    w = workloads.fcc_column(144, 48, 48, 0.7, 24.0, 8.55, jitter=0.01, seed=8, period=30)
    w.fixed = np.ones(len(w.R), np.uint8)
    w.probe_x = 40
    return lbmdem.Sim.from_workload(w, **over)


def _run(calls, **over):
    s = _sim(**over)
    for n in calls:
        s.step(n)
    out, p, c = s.fields(), s.probe(), s.counters()
    assert s.status() == 0 and c["stored"] >= 65536 and c["links"] >= 2 * c["stored"]
    f = s.particles()
    s.close()
    return out, p, f


def test_calls_do_not_show():
    a, pa, fa = _run([37])
    for calls, over in (([1] * 37, {}), ([2, 16, 3, 15, 1], {}), ([5, 32], dict(graph_steps=4)),
                        ([37], dict(monitor_every=3))):
        b, pb, fb = _run(calls, **over)
        assert all(np.array_equal(x, y) for x, y in zip(a, b)), (calls, over)
        assert pa.shape == pb.shape and np.abs(pa - pb).max() <= 1e-13
        for k in ("Fh", "Th"):
            assert np.abs(fa[k] - fb[k]).max() <= 1e-9 * np.abs(fa[k]).max()


def test_segments_do_not_show():
    ref = None
    for every in (40, 16, 2):
        s = _sim()
        got = s.adjoint(40, every, np.full(40, 1 / 3)), s.fields()
        s.close()
        if ref is None:
            ref = got
        assert all(np.array_equal(x, y) for x, y in zip(got[1], ref[1]))
        assert np.abs(got[0][3] - ref[0][3]).max() <= 1e-13
        for x, y in zip(got[0][:3], ref[0][:3]):
            assert abs(x - y) <= 1e-8 * abs(y)
