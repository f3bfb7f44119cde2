"""Launches whose parts are clusters: every block has exactly one part, the parts of an item are one cluster
in order, and together they are the item."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    cxx = os.environ.get("CXX") or shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    cuda = next((d for d in ("/usr/local/cuda/include", os.path.join(os.environ.get("CUDA_HOME", ""), "include"))
                 if os.path.exists(os.path.join(d, "cuda_runtime.h"))), None)
    if cuda is None:
        pytest.skip("no CUDA headers")
    exe = str(tmp_path_factory.mktemp("plan") / "cluster_plan")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2609_32518_b200", "csrc"), "-I",
                    os.path.join(ROOT, "include"), "-I", cuda, os.path.join(HERE, "cluster_plan.cpp"), "-o", exe], check=True)
    return lambda *a: [[int(x) for x in line.split()] for line in subprocess.run(
        [exe, *map(str, a)], check=True, capture_output=True, text=True).stdout.splitlines()]


@pytest.mark.parametrize("heads,grid,chunk,frames,start,parts", [
    (25, (9, 15), 2, 10, 8, 2), (20, (9, 15), 2, 8, 6, 3), (15, (9, 15), 2, 7, 5, 4), (11, (9, 15), 2, 9, 7, 5),
    (10, (9, 15), 2, 11, 9, 6), (6, (9, 15), 2, 6, 4, 7), (7, (9, 15), 2, 7, 5, 8), (2, (8, 8), 2, 6, 4, 6),
    (1, (8, 8), 1, 2, 1, 0), (2, (30, 52), 3, 21, 18, 0), (12, (30, 52), 3, 3, 0, 0)])
def test_every_block_has_one_part(plan, heads, grid, chunk, frames, start, parts):
    (cluster, n, workers), *segs = plan(heads, *grid, chunk, frames, start)
    assert cluster == (parts > 0)
    if not cluster:
        return
    assert n == parts and [s[0] for s in segs] == list(range(workers)) and workers <= 148
    pairs = ((grid[0] * grid[1] * chunk + 127) // 128 + 1) // 2
    assert workers == heads * pairs * parts
    for first in range(0, workers, parts):
        group = segs[first:first + parts]
        assert len({tuple(s[1:3]) for s in group}) == 1
        assert [s[3] for s in group] == [0] + [s[4] for s in group[:-1]] and group[-1][4] == group[0][5]
        assert all(s[3] < s[4] for s in group)
