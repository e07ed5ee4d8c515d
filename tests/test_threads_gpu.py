"""Host threads that each make and pack a context of their own, at the same
time and as the first thing their process does on the GPU, get what one thread
after another gets.  Spheres alone, whose steps are deterministic; one CTA,
several, and a launch per substep."""
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

PROGRAM = """
import sys, threading
import numpy as np
sys.path.insert(0, ".")
import workloads
from paper_1808_08921_gb300 import lbmdem

lbmdem.load()
COUNTS = (40, 300, 1500, 2100)

def run(n, start=None):
    side = int(np.ceil(n ** (1 / 3)))
    X = 4.0 + 5.99 * np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    V = np.random.default_rng(n).uniform(-1e-3, 1e-3, X.shape)
    L = 6 * side + 2
    w = workloads.Workload(name="dry", nx=L, ny=L, nz=L, tau=0.8, X=X, R=np.full(n, 3.0), V=V,
                           fixed=np.zeros(n, np.uint8), dem_substeps=4)
    p = lbmdem.params_from_workload(w, lbm_on=0)
    if start:
        start.wait()
    s = lbmdem.Sim(p)
    s.set_packing(w.X, w.R, w.V, None, w.fixed)
    s.step(20)
    assert s.status() == 0
    out = s.particles()
    s.close()
    return out

start, got = threading.Barrier(2 * len(COUNTS)), {}
def work(k, n):
    got[k] = run(n, start)
threads = [threading.Thread(target=work, args=(k, n)) for k, n in enumerate(2 * COUNTS)]
for t in threads: t.start()
for t in threads: t.join()
for k, n in enumerate(2 * COUNTS):
    ref = run(n)
    assert ref["V"].any() and all(np.array_equal(got[k][q], ref[q]) for q in ref), n
print("same")
"""


def test_contexts_packed_at_the_same_time():
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stdout + r.stderr
