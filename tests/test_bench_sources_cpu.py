"""The bench's DRAM figures hold for the kernel sources they were taken on: every
file the force and density passes are compiled from counts."""
import os
import shutil

import pytest

import bench


def test_sources_follow_the_includes():
    assert sorted(bench._kernel_sources("sph_physics.cu")) == ["sph_boids.cuh", "sph_internal.cuh", "sph_physics.cu"]


@pytest.mark.parametrize("name", ["sph_boids.cuh", "sph_internal.cuh", "sph_physics.cu"])
def test_a_change_of_any_source_changes_the_hash(name, tmp_path, monkeypatch):
    copy = tmp_path / "csrc"
    shutil.copytree(bench.CSRC, copy)
    monkeypatch.setattr(bench, "CSRC", str(copy))
    before = bench._source_sha(*bench._kernel_sources("sph_physics.cu"))
    with open(os.path.join(copy, name), "a") as f:
        f.write("// moved\n")
    assert bench._source_sha(*bench._kernel_sources("sph_physics.cu")) != before
