"""The attention kernel hands P over through named barriers, which have no bounded wait: whatever wait
gave up where, every warp must get past all of them.  A model of the barriers' counts walks through all
orders, with the kernel's own rule (csrc/handover.h) and with two rules that leave a warp behind."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_32518_b200", "csrc")


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    cxx = os.environ.get("CXX") or shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path_factory.mktemp("model") / "hand_over_model")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "hand_over_model.cpp"), "-o", exe],
                   check=True)
    return exe


@pytest.mark.parametrize("tiles,segment", [(1, 1), (2, 1), (2, 2), (3, 2), (4, 4), (5, 2), (5, 5)])
def test_no_order_leaves_a_warp_at_a_barrier(model, tiles, segment):
    out = subprocess.run([model, str(tiles), str(segment)], check=True, capture_output=True, text=True).stdout
    blocked = {line.split()[0]: int(line.split()[2]) for line in out.splitlines()}
    assert blocked["kernel"] == 0
    if tiles > 1:
        assert blocked["one_barrier_arrive"] > 0 and blocked["one_barrier_wait"] > 0
