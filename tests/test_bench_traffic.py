"""bench.py's recorded DRAM traffic: it is the chains' own, and only for the source that it was captured with."""
import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_2004_10892_gb300", "csrc")


@pytest.mark.parametrize("name,text", [
    ("pair.cu", "k_pair("), ("pair.cuh", "PAIR_SMEM_TWO = 98"), ("device_util.cuh", "fmaf(a.x"),
    ("runtime.cu", "PAIR_TILES = 5"), ("runtime.cu", "PAIR_GEMM_PADDING = 16"), ("runtime.cu", "pair_step(one,"),
    ("runtime.cu", "GTPB"),
])
def test_a_change_of_the_chains_drops_the_figure(tmp_path, monkeypatch, name, text):
    here = bench.kernel_source_sha1()
    shutil.copytree(os.path.join(bench.ROOT, CSRC), tmp_path / CSRC)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_source_sha1() == here
    path = tmp_path / CSRC / name
    old = path.read_text()
    assert text in old
    path.write_text(old.replace(text, text + " "))
    assert bench.kernel_source_sha1() != here

