"""The allocators of a search's device pieces (host check of csrc/pieces.h): the
planning kernel reads the windows and costs in 16-byte vectors, so a piece holds
the whole vector of its last element, whatever the number of spectra."""
import os
import shutil
import subprocess

import pytest

from test_sanitize_host import cuda_root

ROOT = os.path.abspath(os.path.join(os.path.dirname(__file__), ".."))


def test_pieces_hold_whole_vectors(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = tmp_path / "pieces_check"
    subprocess.run([cxx, "-O1", "-std=c++17", "-Wall", "-I", os.path.join(cuda_root(), "include"),
                    "-I", os.path.join(ROOT, "paper_2102_02286_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "pieces_check.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.strip() == "ok"
