"""Launches whose work split the GPU tests rely on.  The split of each is pinned on the CPU for a B200 of 148 SMs
(test_attn_plan.py); the GPU tests ask the device for its own limits and check the form where they depend on it."""

import paper_2609_32518_b200 as U

CLUSTERS = [0, 0, 74, 45, 33, 26, 22, 15, 15]   # clusters of n blocks that the 148 SMs of a B200 run at once


def forms(segs):
    """What the segments of a launch are: "whole" items, parts of a "cluster", parts merged through "scratch"."""
    return {"whole" if s[8] == 1 else "cluster" if s[9] == -1 else "scratch" for s in segs}


def shortest_part(segs):
    return min(s[6] - s[5] for s in segs if s[8] > 1)


def split_on_device(shape, starts, window, sink=0, sink_attend=0):
    """The segments of the launch on the current device (a U.Shape)."""
    return U.window_attn_plan(shape, list(starts), window, U.attn_workers()[0], sink, sink_attend, U.attn_clusters())


# name -> (batch, heads, grid, chunk frames, ring frames = window, starts), forms, largest number of parts.
# The first six do not depend on which clusters a device runs, or hardly: behind whole rounds, with more items than
# clusters of two, and with few items of very many tiles there are none; 49 x 3 and 37 x 4 blocks would
# have to fill 147 and all 148 SMs.
SPLITS = {
    "whole_and_parts": ((1, 150, (10, 20), 1, 9, (8,)), {"whole", "scratch"}, 3),        # 15 tiles, the last of 8 keys
    "shares": ((1, 80, (10, 15), 1, 17, (16,)), {"scratch"}, 3),                         # 20 tiles, the last of 118
    "many_parts": ((2, 2, (16, 16), 1, 160, (159, 99)), {"scratch"}, 16),                # 320 and 200 tiles
    "three_parts": ((1, 49, (9, 15), 1, 14, (13,)), {"scratch"}, 3),                     # 15 tiles
    "four_parts": ((1, 37, (9, 15), 1, 40, (39,)), {"scratch"}, 4),                      # 43 tiles
    "shares_of_32_streams": ((33, 5, (8, 20), 1, 3, tuple(2 + b % 3 for b in range(33))), {"whole", "scratch"}, 2),
    "cluster": ((1, 7, (10, 20), 1, 18, (17,)), {"cluster"}, 8),                         # 29 tiles, 3 or 4 a part
}

# batch, heads, grid, chunk frames, ring, window, history, starts, parts of every item
EQUAL_PARTS = [
    (2, 5, (17, 23), 2, 7, 5, ((4, 6, 8, 10), (2, 4, 6)), (12, 8), 3),        # 16 and 17 key tiles
    (1, 1, (20, 30), 3, 9, 9, ((3, 6, 9),), (12,), 8),
    (3, 1, (11, 13), 3, 9, 9, ((), (0, 3), (3, 6, 9)), (0, 6, 12), 4),        # 4 and 11 key tiles
    (2, 4, (16, 24), 1, 6, 6, (tuple(range(3, 9)), (0,)), (9, 1), 6),         # a lone query tile
    (1, 3, (9, 14), 1, 5, 5, ((1, 2, 3, 4, 5),), (6,), 5),                    # frames below a tile
]
