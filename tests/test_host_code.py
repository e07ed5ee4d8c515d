"""Host code of the library on its own, compiled with the host compiler: no
GPU and no CUDA runtime library behind it."""
import os
import shutil
import subprocess

import pytest

from paper_1808_08921_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def _run(name, tmp_path):
    cxx = shutil.which("g++")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    if cxx is None or not os.path.exists(os.path.join(include, "cuda_runtime_api.h")):
        pytest.skip("no host compiler or no CUDA headers")
    exe = str(tmp_path / name)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I" + build.CSRC, "-I" + include,
                    os.path.join(HERE, "host", name + ".cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_arrays_after_a_refused_allocation(tmp_path):
    _run("device_memory", tmp_path)


def test_threads_agree_on_a_device(tmp_path):
    _run("per_device", tmp_path)
