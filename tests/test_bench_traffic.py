"""The DRAM traffic that the benchmark prints is of a capture; it must go when the code changes."""
import os
import shutil

import pytest

import bench


@pytest.mark.parametrize("key", sorted(bench.NCU_TRAFFIC))
def test_a_traffic_figure_goes_when_a_source_that_decides_it_changes(key, tmp_path, monkeypatch):
    csrc = os.path.join("paper_2404_14469_b200", "csrc")
    shutil.copytree(os.path.join(bench.ROOT, csrc), tmp_path / csrc)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    nbytes, sources, _ = bench.NCU_TRAFFIC[key]
    monkeypatch.setitem(bench.NCU_TRAFFIC, key, (nbytes, sources, bench.sources_digest(sources)))
    for src in sources:
        path = tmp_path / csrc / src
        whole = path.read_bytes()
        assert bench.ncu_traffic(*key) == nbytes
        path.write_bytes(whole + b"\n")
        assert bench.ncu_traffic(*key) is None
        path.write_bytes(whole)


def test_the_scoring_plan_is_among_them():
    # wave size and lag are set there
    assert {"score_kernel.cuh", "snapkv_score.cu", "snapkv_internal.h"} <= set(bench.NCU_TRAFFIC["score", 2][1])
