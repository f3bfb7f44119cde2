"""The work split of the attention kernel, replayed on the host (no GPU).

The kernel's roles all walk the same integer schedule; `unstep_window_attn_plan(_clusters)` lists it with the
same code compiled for the host.  Whatever the shape, window and worker count, every (item, key
tile) step must be covered exactly once, a split item's parts must be counted correctly (a part
that waits for more parts than exist would never merge, and its rows would never be written), and
no two parts of one worker may share a scratch slot.  Parts that are a cluster take no slot: they are one
segment per worker, and the parts of an item the blocks of one cluster, in order."""

import ctypes
import itertools

import pytest

import paper_2609_32518_b200 as U
from splits import CLUSTERS, EQUAL_PARTS, SPLITS, forms


def check_plan(shape, starts, window, workers, sink=0, sink_attend=0, clusters=None):
    segs = U.window_attn_plan(shape, starts, window, workers, sink, sink_attend, clusters)
    in_cluster = any(s[8] > 1 and s[9] == -1 for s in segs)
    assert clusters is not None or not in_cluster
    T = shape.grid_h * shape.grid_w
    q_tiles = -(-shape.chunk_frames * T // 128)
    q_pairs = (q_tiles + 1) // 2
    covered = {}
    parts_seen = {}
    slots_of_worker = {}
    for (w, b, h, qp, nq, t0, t1, tiles, parts, slot) in segs:
        assert 0 <= w < workers and 0 <= b < shape.batch and 0 <= h < shape.heads and 0 <= qp < q_pairs
        assert nq == (2 if 2 * qp + 1 < q_tiles else 1)
        assert 0 <= t0 < t1 <= tiles
        item = (b, h, qp)
        for t in range(t0, t1):
            assert (item, t) not in covered, f"step {(item, t)} given to two workers"
            covered[(item, t)] = w
        whole = t0 == 0 and t1 == tiles
        assert (parts == 1 and slot == -1) if whole else (parts >= 2 and slot in ((-1,) if in_cluster else (0, 1)))
        if in_cluster:
            assert parts == segs[0][8] and t1 - t0 in (tiles // parts, tiles // parts + 1)
            parts_seen.setdefault(item, []).append((w, parts))
        elif not whole:
            parts_seen.setdefault(item, []).append((w, parts))
            assert slot not in slots_of_worker.setdefault(w, set()), f"worker {w} reuses scratch slot {slot}"
            slots_of_worker[w].add(slot)
    # every step of every item exactly once
    n_items = shape.batch * shape.heads * q_pairs
    items = {k[0] for k in covered}
    assert len(items) == n_items
    by_item = {}
    for (item, t) in covered:
        by_item.setdefault(item, set()).add(t)
    tiles_of = {}
    for (w, b, h, qp, nq, t0, t1, tiles, parts, slot) in segs:
        tiles_of[(b, h, qp)] = tiles
    for item, ts in by_item.items():
        assert ts == set(range(tiles_of[item])), f"item {item}: steps missing"
    # a split item: as many parts as each of its parts expects, on consecutive workers
    for item, lst in parts_seen.items():
        ws = sorted(w for w, _ in lst)
        assert all(n == len(lst) for _, n in lst), f"item {item}: {len(lst)} parts, expected {[n for _, n in lst]}"
        assert ws == list(range(ws[0], ws[0] + len(ws)))
        if in_cluster:   # the blocks of a cluster are neighbours from a multiple of its size on, its parts in their order
            assert ws[0] % len(ws) == 0
            assert [s[5] for s in segs if (s[1], s[2], s[3]) == item] == sorted(s[5] for s in segs if (s[1], s[2], s[3]) == item)
    if in_cluster:
        parts = segs[0][8]
        assert [s[0] for s in segs] == list(range(n_items * parts))
        assert n_items <= clusters[parts] - (3 if parts in (3, 5) else 0)   # room for odd ones
    return segs


def test_shapes_whose_remainder_is_smaller_than_the_grid():
    # 10 heads x 15 query pairs = 150 items on 148 workers: one whole round, then 2 items x 30
    # tiles = 60 steps for 148 workers
    sh = U.Shape.make(batch=1, heads=10, chunk_frames=3, grid_h=32, grid_w=40, ring_frames=3)
    segs = check_plan(sh, [0], 3, 148)
    assert max(s[0] for s in segs) == 147
    # 11 heads of one query tile, 2 key tiles in all: the launch shrinks to very few workers
    sh = U.Shape.make(batch=1, heads=11, chunk_frames=2, grid_h=8, grid_w=8, ring_frames=2)
    check_plan(sh, [0], 2, 148)


def test_the_1p3b_and_14b_shapes_on_148_and_74_workers():
    sh = U.Shape.make(batch=1, heads=12, chunk_frames=3, grid_h=30, grid_w=52, ring_frames=21)
    for workers in (148, 74):
        segs = check_plan(sh, [18], 21, workers)
        assert sum(s[6] - s[5] for s in segs) == 12 * 19 * 256
    sh5 = U.Shape.make(batch=1, heads=40, chunk_frames=3, grid_h=45, grid_w=80, ring_frames=12)
    check_plan(sh5, [9], 12, 148)
    sh4 = U.Shape.make(batch=4, heads=12, chunk_frames=3, grid_h=30, grid_w=52, ring_frames=21)
    check_plan(sh4, [0, 6, 12, 18], 21, 148)


@pytest.mark.parametrize("workers", [1, 2, 5, 31, 74, 148])
def test_sweep_of_small_shapes(workers):
    for heads, (gh, gw), fc, win in itertools.product((1, 2, 3, 10, 11), ((8, 8), (8, 25), (3, 5), (16, 20)),
                                                      (1, 2, 3), (0, 1, 4)):
        ring = fc + win
        sh = U.Shape.make(batch=2, heads=heads, chunk_frames=fc, grid_h=gh, grid_w=gw, ring_frames=ring)
        check_plan(sh, [ring + 1, 0], ring, workers)


def test_sink_prefix_and_bad_arguments():
    sh = U.Shape.make(batch=1, heads=12, chunk_frames=3, grid_h=30, grid_w=52, ring_frames=6)
    segs = check_plan(sh, [18], 6, 148, sink=3, sink_attend=3)
    # frames 0..2 sit in slots 0..2 and frames 15..20 in slots 3..8: one run of 14040 keys
    assert segs[0][7] == -(-9 * 1560 // 128)
    # a chunk later the ring has wrapped: frames 18..20 in slots 6..8, 21..23 in slots 3..5 -> runs 0..2 | 6..8 | 3..5
    segs = check_plan(sh, [21], 6, 148, sink=3, sink_attend=3)
    assert segs[0][7] == 3 * -(-3 * 1560 // 128)
    with pytest.raises(U.UnstepError):
        U.window_attn_plan(sh, [18], 7, 148)          # window longer than the ring
    with pytest.raises(U.UnstepError):
        U.window_attn_plan(sh, [18], 6, 0)            # no workers


def test_launches_smaller_than_the_grid_cut_every_item_into_equal_parts():
    # (batch, heads, grid, chunk frames, ring, window, starts) -> parts of every item
    for b, heads, grid, fc, ring, win, starts, parts in [
            (2, 5, (17, 23), 2, 7, 5, [12, 8], 3),     # items of 16 and of 17 key tiles
            (1, 1, (20, 30), 3, 9, 9, [12], 5),
            (3, 1, (11, 13), 3, 9, 9, [0, 6, 12], 3),  # items of 4 and of 11 key tiles
            (1, 3, (9, 14), 1, 5, 5, [6], 1)]:         # whole items
        sh = U.Shape.make(batch=b, heads=heads, chunk_frames=fc, grid_h=grid[0], grid_w=grid[1], ring_frames=ring)
        segs = check_plan(sh, starts, win, 148)
        assert {s[8] for s in segs} == {parts}
        assert len(segs) == 1 + max(s[0] for s in segs)   # one segment per worker
        for s in segs:
            assert abs((s[6] - s[5]) - s[7] / parts) < 1


def test_split_of_more_steps_than_32_bit_products_hold():
    # 32 items of 8.4 million key tiles: shares across items in 64-bit arithmetic
    frames = 262143
    sh = U.Shape.make(batch=1, heads=2, chunk_frames=1, grid_h=64, grid_w=64, ring_frames=frames)
    segs = U.window_attn_plan(sh, [frames - 1], frames, 148)
    tiles = frames * 64 * 64 // 128
    items = {}
    for (w, b, h, qp, nq, t0, t1, n, parts, slot) in segs:
        assert n == tiles and 0 <= t0 < t1 <= tiles
        items.setdefault((h, qp), []).append((t0, t1, w, parts))
    assert len(items) == 2 * 16
    total = len(items) * tiles
    for spans in items.values():
        spans.sort()
        assert [s[0] for s in spans] == [0] + [s[1] for s in spans[:-1]] and spans[-1][1] == tiles
        assert all(s[3] == len(spans) for s in spans)
        assert [s[2] for s in spans] == list(range(spans[0][2], spans[0][2] + len(spans)))
    work = {}
    for s in segs:
        work[s[0]] = work.get(s[0], 0) + s[6] - s[5]
    assert len(work) == 148 and max(work.values()) - min(work.values()) <= 1 and sum(work.values()) == total


@pytest.mark.parametrize("frames", [14_510_024, 14_510_025, 14_600_000, 1 << 24, 1 << 29])
def test_parts_of_items_of_many_tiles(frames):
    # frames of one token, a key tile each: tiles x 148 parts passes 2^31 between the first two, and the
    # item is cut in 64-bit arithmetic from there on
    sh = U.Shape.make(batch=1, heads=1, chunk_frames=1, grid_h=1, grid_w=1, ring_frames=frames)
    segs = U.window_attn_plan(sh, [frames - 1], frames, 148)
    assert [s[0] for s in segs] == list(range(148)) and {s[8] for s in segs} == {148}
    assert [s[5] for s in segs] == [0] + [s[6] for s in segs[:-1]] and segs[-1][6] == frames
    assert {s[6] - s[5] for s in segs} <= {frames // 148, frames // 148 + 1}


def test_workers_rise_and_fall_along_a_clip_within_the_grid():
    # scratch has two slots for each of the grid's workers, whatever the start frame
    workers = {}
    for heads, fc, starts in [(3, 3, (0, 3, 18)), (1, 1, (0, 18, 19, 20))]:
        sh = U.Shape.make(batch=1, heads=heads, chunk_frames=fc, grid_h=30, grid_w=52, ring_frames=21)
        for start in starts:
            segs = check_plan(sh, [start], 21, 148)
            workers[heads, start] = 1 + max(s[0] for s in segs)
    assert workers[3, 0] < workers[3, 3] and workers[1, 20] < workers[1, 19]
    assert max(workers.values()) <= 148


def test_sweep_of_small_shapes_on_a_device_that_runs_clusters():
    # two streams at different fill levels, without and with sink frames
    seen = {}
    for heads, (gh, gw), fc, win, sink in itertools.product((1, 2, 7, 25, 50, 80), ((8, 8), (3, 5), (9, 15), (16, 20)),
                                                            (1, 3), (0, 6), (0, 2)):
        ring = fc + win
        sh = U.Shape.make(batch=2, heads=heads, chunk_frames=fc, grid_h=gh, grid_w=gw, ring_frames=ring)
        segs = check_plan(sh, [ring + 3, 0], ring, 148, sink, sink, CLUSTERS)
        for f in forms(segs):
            seen.setdefault(f, set()).add(max(s[8] for s in segs))
    assert seen["cluster"] >= {2, 3, 4, 5, 6, 8} and "whole" in seen and len(seen["scratch"]) > 1


def test_limits_of_the_device_decide_which_clusters_a_launch_has():
    sh = U.Shape.make(batch=1, heads=8, chunk_frames=2, grid_h=9, grid_w=15, ring_frames=9)   # 16 items of 10 tiles
    parts = lambda clusters: {s[8] for s in check_plan(sh, [7], 9, 148, clusters=clusters)}   # noqa: E731
    assert parts(CLUSTERS) == {5} and parts([0] * 6 + [0, 0, 16]) == {8}
    none = check_plan(sh, [7], 9, 148, clusters=[0] * 9)
    assert none == check_plan(sh, [7], 9, 148) and {s[9] for s in none} == {0}
    # no clusters behind whole rounds, nor of more parts than the shortest stream has tiles
    sh = U.Shape.make(batch=1, heads=150, chunk_frames=1, grid_h=10, grid_w=20, ring_frames=9)
    assert forms(check_plan(sh, [8], 9, 148, clusters=CLUSTERS)) == {"whole", "scratch"}
    sh = U.Shape.make(batch=2, heads=1, chunk_frames=1, grid_h=8, grid_w=8, ring_frames=9)
    assert {s[8] for s in check_plan(sh, [8, 2], 9, 148, clusters=CLUSTERS)} == {3}


@pytest.mark.parametrize("parts,most", [(3, 42), (5, 23)])
def test_clusters_of_odd_size_leave_room(parts, most):
    # 13 key tiles; with all 45 clusters of 3, or 26 of 5, a launch under the one before it ran in two waves
    # (15 of 7 are 105 blocks and never did)
    for items in range(most - 2, CLUSTERS[parts] + 1):
        sh = U.Shape.make(batch=1, heads=items, chunk_frames=2, grid_h=8, grid_w=15, ring_frames=13)
        segs = check_plan(sh, [11], 13, 148, clusters=CLUSTERS)
        assert (forms(segs) == {"cluster"} and segs[0][8] == parts) == (items <= most), items
    sh = U.Shape.make(batch=1, heads=15, chunk_frames=2, grid_h=8, grid_w=15, ring_frames=13)
    assert {s[8] for s in check_plan(sh, [11], 13, 148, clusters=CLUSTERS)} == {7}


@pytest.mark.parametrize("heads,grid,fc,ring,form,parts", [
    (74, (10, 20), 1, 2, "whole", 1), (33, (10, 20), 1, 2, "whole", 1), (41, (8, 8), 2, 3, "whole", 1),   # 4, 4, 3 tiles
    (2, (8, 8), 2, 6, "cluster", 6), (5, (17, 23), 2, 13, "cluster", 6),                # 2 items of 6 tiles, 20 of 40
    (10, (17, 23), 2, 5, "cluster", 3), (13, (17, 23), 2, 13, "cluster", 2),            # 40 items of 16 tiles, 52 of 40
    (10, (30, 52), 1, 15, "scratch", 2), (16, (17, 23), 2, 21, "scratch", 2)])          # 70 items of 183 tiles, 64 of 65
def test_the_split_is_the_one_that_was_measured_to_be_shortest(heads, grid, fc, ring, form, parts):
    sh = U.Shape.make(batch=1, heads=heads, chunk_frames=fc, grid_h=grid[0], grid_w=grid[1], ring_frames=ring)
    segs = check_plan(sh, [ring - fc], ring, 148, clusters=CLUSTERS)
    assert forms(segs) == {form} and max(s[8] for s in segs) == parts


def test_the_list_without_clusters_and_its_arguments():
    sh = U.Shape.make(batch=1, heads=8, chunk_frames=2, grid_h=9, grid_w=15, ring_frames=9)
    want = [x for s in U.window_attn_plan(sh, [7], 9, 148) for x in s]
    buf, n, start = (ctypes.c_int32 * len(want))(), ctypes.c_int32(0), (ctypes.c_int32 * 1)(7)
    rc = U.lib().unstep_window_attn_plan(ctypes.byref(sh), 0, start, 9, 0, 148, buf, len(want) // 10, ctypes.byref(n))
    assert rc == 0 and 10 * n.value == len(want) and list(buf) == want
    with pytest.raises(ValueError):
        U.window_attn_plan(sh, [7], 9, 148, clusters=[0, 0, 74])
    assert U.lib().unstep_attn_clusters(None) == -1


@pytest.mark.parametrize("name", list(SPLITS))
def test_launches_that_the_gpu_tests_rely_on(name):
    (batch, heads, grid, fc, ring, starts), want, parts = SPLITS[name]
    sh = U.Shape.make(batch=batch, heads=heads, chunk_frames=fc, grid_h=grid[0], grid_w=grid[1], ring_frames=ring)
    segs = U.window_attn_plan(sh, starts, ring, 148, clusters=CLUSTERS)
    assert forms(segs) == want and max(s[8] for s in segs) == parts
    if batch <= 32:
        check_plan(sh, starts, ring, 148, clusters=CLUSTERS)


@pytest.mark.parametrize("batch,heads,grid,fc,ring,win,history,starts,parts", EQUAL_PARTS)
def test_launches_of_equal_parts_are_clusters(batch, heads, grid, fc, ring, win, history, starts, parts):
    sh = U.Shape.make(batch=batch, heads=heads, chunk_frames=fc, grid_h=grid[0], grid_w=grid[1], ring_frames=ring)
    segs = check_plan(sh, starts, win, 148, clusters=CLUSTERS)
    assert forms(segs) == {"cluster"} and {s[8] for s in segs} == {parts}
