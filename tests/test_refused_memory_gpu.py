"""Calls that are refused memory, at each of their allocations in turn: the
call returns OOM, nothing runs on the context until it has a packing again,
and a smaller packing on it then gives what a new context gives.  No memory has
to run out: a preloaded cudaMalloc asks for more than there can be."""
import os
import shutil
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

PROGRAM = """
import ctypes, sys
import numpy as np
sys.path.insert(0, ".")
import workloads
from paper_1808_08921_gb300 import lbmdem

OOM, STATE = -2, -6
lib = lbmdem.load()
shim = ctypes.CDLL(sys.argv[1])
allowed, refused = ctypes.c_long.in_dll(shim, "allowed"), ctypes.c_long.in_dll(shim, "refused")

def work(n, R):
    w = workloads.random_small(3, nx=60, ny=30, nz=30, n=n, R=R, vel=0.01)
    w.amplitude, w.omega, w.body_force = 1e-3, 0.2, (1e-4, 0.0, 0.0)
    return w

small, large = work(5, 3.0), work(60, 2.6)

def pack(s, w):
    s.set_packing(w.X, w.R, w.V, w.W, w.fixed)

def sim(w):
    return lbmdem.Sim.from_workload(w, skin=0.5, dem_skin=1.0)

def outputs(s):
    s.step(21)
    assert s.status() == 0
    return s.fields() + (s.particles()["X"],)

def code(f, *a):
    try:
        f(*a)
        return 0
    except lbmdem.LbmDemError as e:
        return e.code

r = sim(small)
ref = outputs(r)
r.close()

def attempt(k, call):
    s = sim(small)
    s.step(4)
    batch = lbmdem.Batch([s])
    allowed.value = k
    got = code(call, s)
    allowed.value = -1
    if got:
        assert got == OOM, got
        for f in (lambda: s.step(2), s.fields, s.plane_means, s.particles, s.relayout, lambda: batch.step([2])):
            assert code(f) == STATE
        pack(s, small)
    else:
        pack(s, small)
    out = outputs(s)
    batch.close()
    s.close()
    assert np.array_equal(out[2], ref[2])
    assert np.abs(out[0] - ref[0]).max() <= 1e-7 and np.abs(out[1] - ref[1]).max() <= 2e-6 * np.abs(ref[1]).max()
    assert np.abs(out[3] - ref[3]).max() <= 1e-9
    return got

call = dict(set_packing=lambda s: pack(s, large), relayout=lambda s: s.relayout())[sys.argv[2]]
k = 0
while attempt(k, call) == OOM:
    k += 1
    assert k < 200
assert refused.value >= k > 0
print("refused at each of", k, "allocations")
print("usable")
"""


@pytest.mark.parametrize("call", ["set_packing", "relayout"])
def test_every_allocation_refused_in_turn(call, tmp_path):
    cc, shim = shutil.which("gcc"), str(tmp_path / "refuse_alloc.so")
    subprocess.run([cc, "-shared", "-fPIC", "-O1", os.path.join(ROOT, "tests", "host", "refuse_alloc.c"), "-o", shim,
                    "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", PROGRAM, shim, call], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, LD_PRELOAD=shim))
    assert r.returncode == 0 and "usable" in r.stdout, r.stdout + r.stderr
    print(r.stdout)
