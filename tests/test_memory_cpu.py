"""The host code when device memory runs out: a call that fails for lack of memory leaves the handle so that the same
call works once there is memory, and every buffer that a launch uses is there and large enough.

The library's host sources are compiled with a stand-in for the CUDA runtime and the kernel launchers
(fake_device.cpp); no GPU is used.  Each scenario refuses the n-th allocation of a call and all after it, for every n.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1605_04521_gb300", "csrc")
SOURCES = ["api.cpp", "host_setup.cpp", "fronts_plan.cpp", "fronts_weak.cpp", "tables.cpp", "dense.cpp", "block_fgmres.cpp", "gcrodr.cpp"]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(nvcc):
        pytest.skip("no C++ compiler or no CUDA headers")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    out = str(tmp_path_factory.mktemp("fake") / "fake_device")
    src = [os.path.join(CSRC, f) for f in SOURCES] + [os.path.join(ROOT, "tests", "fake_device.cpp")]
    objs = [out + f".{i}.o" for i in range(len(src))]
    jobs = [subprocess.Popen([cxx, "-std=c++17", "-O1", "-fno-pie", "-pthread", "-I", CSRC, "-I", cuda, "-c", s, "-o", o],
                             stderr=subprocess.PIPE, text=True) for s, o in zip(src, objs)]
    for j in jobs:
        err = j.communicate()[1]
        assert j.returncode == 0, err
    # launchers that no scenario reaches are left undefined
    r = subprocess.run([cxx, "-no-pie", "-pthread", "-Wl,--unresolved-symbols=ignore-all", *objs, "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


def findings(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=300)
    return r.returncode, r.stdout


@pytest.mark.parametrize("scenario", ["factor32", "factor64", "factor_dense", "factor_weak32", "factor_weak64"])
def test_factor_again_after_running_out_of_memory(program, scenario):
    assert findings(program, scenario) == (0, "")


@pytest.mark.parametrize("scenario", ["solve32", "solve64"])
def test_solve_again_after_running_out_of_memory(program, scenario):
    """A solve of three columns runs out of memory after one of two: then two and three columns again."""
    assert findings(program, scenario) == (0, "")


@pytest.mark.parametrize("scenario", ["setup", "setup_dense"])
def test_failed_set_up_leaves_no_memory_behind(program, scenario):
    assert findings(program, scenario) == (0, "")


@pytest.mark.parametrize("scenario", ["delay1", "delay2", "delay3", "always_weak"])
def test_trees_with_unknowns_moved_up(program, scenario):
    """Random unknowns eliminated later than planned: every unknown once, every coupling inside a front, borders and
    sources consistent."""
    assert findings(program, scenario) == (0, "")
