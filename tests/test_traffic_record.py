"""The key of the recorded DRAM traffic (bench.search_source_hash) changes with
every source that decides how many bytes the search kernel moves."""
import os
import shutil

import bench


def test_key_covers_what_decides_the_traffic(tmp_path, monkeypatch):
    csrc = os.path.join("paper_2102_02286_gb300", "csrc")
    shutil.copytree(os.path.join(bench.ROOT, csrc), tmp_path / csrc)
    key = bench.search_source_hash()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.search_source_hash() == key
    # the kernel, the units it is given (planner and costs), its launch shape and shared memory, the index
    for name in ("search_kernel.cuh", "search_kernels.cuh", "search.cu", "hicops_internal.h", "index_build.cu"):
        path = tmp_path / csrc / name
        text = path.read_text()
        path.write_text(text + "// changed\n")
        assert bench.search_source_hash() != key, name
        path.write_text(text)
