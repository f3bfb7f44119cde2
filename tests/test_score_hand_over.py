"""S goes back to the Q K^T issuer and P on to the P V issuer through named barriers, which have no bounded
wait: whatever wait gave up where, every warp must get past all of them.  A model of the barriers' counts
walks through all orders, with the kernel's own rule (csrc/handover.h) and with rules that leave somebody behind: one
barrier of each kind, and warps that gave up and do not wait at the barriers."""

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
    exe = str(tmp_path_factory.mktemp("model") / "score_hand_over_model")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "score_hand_over_model.cpp"), "-o", exe],
                   check=True)
    return exe


# four warps of one group with both issuers, and two groups of fewer warps in turn
@pytest.mark.parametrize("tiles,segment,groups,warps", [(1, 1, 1, 4), (2, 1, 1, 4), (3, 3, 1, 4), (3, 2, 1, 3),
                                                        (4, 2, 1, 2), (5, 5, 1, 2), (2, 2, 2, 2), (2, 1, 2, 2), (3, 3, 2, 1)])
def test_no_order_leaves_a_warp_at_a_barrier(model, tiles, segment, groups, warps):
    out = subprocess.run([model, str(tiles), str(segment), str(groups), str(warps)], check=True, capture_output=True,
                         text=True).stdout
    blocked = {line.split()[0]: int(line.split()[2]) for line in out.splitlines()}
    assert blocked["kernel"] == 0
    if tiles > 1:
        assert blocked["one_barrier_arrive"] > 0
    if tiles > 1 and warps > 1:
        assert blocked["one_barrier"] > 0
    if tiles > 2:
        assert blocked["two_barriers_arrive"] > 0
