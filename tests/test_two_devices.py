"""Indexes on two devices in one process (host check: the library's objects against
tests/fake_runtime.cpp): each device's search kernels are opted into its shared
memory, and grids follow each device's number of SMs."""
import glob
import os
import shutil
import subprocess

import pytest

from paper_2102_02286_gb300 import build as pkg_build

ROOT = os.path.abspath(os.path.join(os.path.dirname(__file__), ".."))


def test_searches_on_two_devices(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    pkg_build.build()
    objects = sorted(glob.glob(os.path.join(pkg_build.BUILD, "*.o")))
    assert len(objects) == len(pkg_build.CU_SOURCES) + len(pkg_build.CPP_SOURCES)
    exe = str(tmp_path / "fake_runtime")
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", pkg_build.INCLUDE,
                    os.path.join(ROOT, "tests", "fake_runtime.cpp"), *objects, "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.strip() == "ok"
