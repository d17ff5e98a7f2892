"""The benchmark's DRAM traffic figure comes from a profile of the gridder, and only while every source that the
gridder is made of is the one that was profiled."""
import os

import pytest

import bench

SOURCES = ["grid.cu", "pairs.cuh", "internal.cuh"]


@pytest.fixture
def root(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_1403_4209_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for name in SOURCES:
        (csrc / name).write_text("// " + name)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "k_grid_wproj_2k.md").write_text(
        "- gridder sources sha256[:16]: `%s`\n- dram bytes per update: `0.25`\n" % bench._gridder_sources_hash())
    return csrc


def test_traffic_of_the_profiled_sources(root):
    assert bench._gridder_traffic(8.0) == 2.0


@pytest.mark.parametrize("name", SOURCES)
def test_no_traffic_after_a_change(root, name):
    (root / name).write_text("// changed")
    assert bench._gridder_traffic(8.0) is None


def test_every_header_of_the_gridder_is_covered():
    csrc = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_1403_4209_gb300", "csrc")
    seen, todo = set(), ["grid.cu"]
    while todo:
        name = todo.pop()
        seen.add(name)
        for line in open(os.path.join(csrc, name)):
            if line.startswith('#include "') and line.split('"')[1] in os.listdir(csrc) and line.split('"')[1] not in seen:
                todo.append(line.split('"')[1])
    assert seen == set(bench.GRIDDER_SOURCES)
