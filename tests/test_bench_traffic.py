"""The bench quotes the committed DRAM traffic only while every source that the measured kernels are compiled from is the
one it was taken on: k_prop.cu, the kernel's body in fwime_prop.cuh and the two-step kernel in k_pair.cu."""
import os
import shutil

import pytest

import bench

SOURCES = ["k_prop.cu", "fwime_prop.cuh", "k_pair.cu"]


@pytest.fixture
def tree(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_2206_02362_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for name in SOURCES:
        shutil.copy(os.path.join(bench.ROOT, "paper_2206_02362_gb300", "csrc", name), csrc / name)
    shutil.copytree(os.path.join(bench.ROOT, "profiles"), tmp_path / "profiles")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    return csrc


def test_traffic_is_of_the_current_kernels(tree):
    t = bench.ncu_traffic()
    assert t is not None
    assert 0.9 < t["dram_bytes_per_launch"] / t["algorithmic_bytes_per_launch"] < 1.2


@pytest.mark.parametrize("name", SOURCES)
def test_traffic_is_dropped_with_any_of_its_sources(tree, name):
    with open(tree / name, "a") as f:
        f.write("\n// changed\n")
    assert bench.ncu_traffic() is None
