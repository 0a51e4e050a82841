"""The library's host side without a GPU: its objects linked with a stand-in for the CUDA
runtime (tests/host/fake_cudart.h) whose launches fail on demand, run by
tests/host/launch_check.cpp in a process of its own.  The programs end by themselves; the
time limit is what fails a host loop that a refused launch leaves without an end."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_1508_04596_gb300 import build
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    objs = [os.path.join(build.OBJ, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    build.build(force=not all(os.path.exists(o) for o in objs))
    exe = str(tmp_path_factory.mktemp("launch") / "launch_check")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-I" + cuda, "-I" + os.path.join(build.ROOT, "include"),
                    os.path.join(HERE, "host", "launch_check.cpp"), *objs, "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("check", ["smoother_levels", "device_loops", "tickets", "refused_sums", "plans"])
def test_host_side(program, check):
    r = subprocess.run([program, check], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
