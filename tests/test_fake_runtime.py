"""Host checks of the library's objects against a runtime of two devices that runs
no kernels (tests/fake_runtime.cpp).  Indexes on two devices in one process: each
device's search kernels are opted into its shared memory, and grids follow its
number of SMs.  The server: requests that fill the pool exactly are taken."""
import glob
import os
import shutil
import subprocess

import pytest

from paper_2102_02286_gb300 import build as pkg_build

ROOT = os.path.abspath(os.path.join(os.path.dirname(__file__), ".."))


@pytest.mark.parametrize("check", ["two_devices", "server_blocks"])
def test_host_side(tmp_path, check):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    pkg_build.build()
    objects = sorted(glob.glob(os.path.join(pkg_build.BUILD, "*.o")))
    assert len(objects) == len(pkg_build.CU_SOURCES) + len(pkg_build.CPP_SOURCES)
    exe = str(tmp_path / "fake_runtime")
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", pkg_build.INCLUDE,
                    os.path.join(ROOT, "tests", "fake_runtime.cpp"), *objects, "-o", exe], check=True)
    out = subprocess.run([exe, check], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.strip() == "ok"
