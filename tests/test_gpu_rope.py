"""GPU parity of the RoPE table and the fused RoPE + ring append against the oracle
(through the C ABI).  Ring contents and q_out must match bit for bit."""

import numpy as np
import pytest
import torch

import oracle as O
import paper_2609_32518_b200 as U
import workloads as W
from harness import (SENTINEL, DevicePath, OraclePath, abi_shape, assert_ring_equal, stream_history,
                     to_bits, to_dev)

pytestmark = pytest.mark.gpu


def ulp_diff(a: np.ndarray, b: np.ndarray) -> np.ndarray:
    ia = a.view(np.int32).astype(np.int64)
    ib = b.view(np.int32).astype(np.int64)
    ia = np.where(ia < 0, -(ia & 0x7FFFFFFF), ia)
    ib = np.where(ib < 0, -(ib & 0x7FFFFFFF), ib)
    return np.abs(ia - ib)


@pytest.mark.parametrize("grid,fc,start", [((8, 8), 2, 0), ((8, 8), 2, 16), ((30, 52), 3, 18),
                                           ((30, 52), 3, 120), ((45, 80), 3, 9), ((5, 7), 1, 3)])
def test_table_matches_oracle_within_one_ulp(grid, fc, start):
    sh = W.Shape(batch=1, heads=1, chunk_frames=fc, grid_h=grid[0], grid_w=grid[1], ring_frames=fc)
    L = sh.chunk_tokens
    cos = torch.empty((L, 64), dtype=torch.float32, device="cuda")
    sin = torch.empty_like(cos)
    U.rope_table(abi_shape(sh), start, cos, sin)
    rc, rs = O.rope_table(start, fc, grid[0], grid[1])
    gc, gs = cos.cpu().numpy(), sin.cpu().numpy()
    # 1 float32 ulp, except next to zero where one ulp of the value is far below the
    # double-precision evaluation error: there the absolute difference is bounded instead
    for g, r in ((gc, rc), (gs, rs)):
        d = ulp_diff(g, r)
        close = (d <= 1) | (np.abs(g.astype(np.float64) - r.astype(np.float64)) < 1e-12)
        assert close.all(), f"{(~close).sum()} table entries differ by more than 1 ulp"
        assert (d == 0).mean() > 0.999
    if start == 0:
        assert (gc[0] == 1.0).all() and (gs[0] == 0.0).all()


@pytest.mark.parametrize("grid,fc,bands", [((1, 1), 1, (44, 42, 42)), ((7, 9), 2, (44, 42, 42)),
                                           ((9, 8), 1, (2, 124, 2)), ((16, 17), 3, (124, 2, 2)),
                                           ((8, 63), 1, (2, 2, 124)), ((2100, 1), 1, (44, 42, 42))])
def test_table_at_the_edges_of_its_tiles_and_with_other_bands(grid, fc, bands):
    # tiles of 8 x 8 tokens, 384 threads: whole tiles, remainders of 1 and 7, bands of one and of 62 pairs
    sh = U.Shape.make(1, 1, fc, grid[0], grid[1], fc, bands=bands, rope_base=500.0)
    cos = torch.full((sh.chunk_tokens, 64), float("nan"), dtype=torch.float32, device="cuda")
    sin = torch.full_like(cos, float("nan"))
    U.rope_table(sh, 5, cos, sin)
    for got, want in zip((cos, sin), O.rope_table(5, fc, grid[0], grid[1], bands, 500.0)):
        g = got.cpu().numpy()
        close = (ulp_diff(g, want) <= 1) | (np.abs(g.astype(np.float64) - want.astype(np.float64)) < 1e-12)
        assert close.all()


def test_cfg1_append_bit_exact_and_sentinels():
    wl = W.WORKLOADS["cfg1"]
    dev, ora = DevicePath(wl.shape), OraclePath(wl.shape)
    stream_history(wl, dev, ora)
    q, k, v = W.batch_qkv(wl, wl.measured_starts)
    q_out = dev.append(wl.measured_starts, q, k, v)
    q_ref = ora.append(wl.measured_starts, q, k, v)
    assert np.array_equal(to_bits(q_out), q_ref)
    assert_ring_equal(dev, ora)
    # every slot was written exactly once: no sentinel is left, V is a bit copy of the input
    assert not (to_bits(dev.ring_k) == SENTINEL).all(axis=-1).any()
    assert np.array_equal(to_bits(dev.ring_v)[0, 4], v[0, :64])


def test_untouched_slots_keep_their_bytes_and_overwrite_is_idempotent():
    wl = W.WORKLOADS["cfg1"]
    dev, ora = DevicePath(wl.shape), OraclePath(wl.shape)
    qa, ka, va = W.batch_qkv(wl, [8], tag=0)          # frames 8, 9 -> slots 2, 3
    qb, kb, vb = W.batch_qkv(wl, [8], tag=1)
    dev.append([8], qa, ka, va)
    ora.append([8], qa, ka, va)
    rk = to_bits(dev.ring_k)
    for slot in (0, 1, 4, 5):
        assert (rk[0, slot] == SENTINEL).all()
    assert_ring_equal(dev, ora)
    dev.append([8], qb, kb, vb)                        # the same chunk again: overwrite
    ora.append([8], qb, kb, vb)
    assert_ring_equal(dev, ora)
    fresh = DevicePath(wl.shape)
    fresh.append([8], qb, kb, vb)
    assert torch.equal(fresh.ring_k.view(torch.int16), dev.ring_k.view(torch.int16))
    assert torch.equal(fresh.ring_v.view(torch.int16), dev.ring_v.view(torch.int16))


def test_wrapped_ring_and_in_place_q():
    wl = W.WORKLOADS["cfg1_wrapped"]
    dev, ora = DevicePath(wl.shape), OraclePath(wl.shape)
    stream_history(wl, dev, ora)
    q, k, v = W.batch_qkv(wl, wl.measured_starts)
    q_out = dev.append(wl.measured_starts, q, k, v, in_place=True)   # q_out aliases q_in
    q_ref = ora.append(wl.measured_starts, q, k, v)
    assert np.array_equal(to_bits(q_out), q_ref)
    assert_ring_equal(dev, ora)


def test_ragged_shape_many_streams_with_own_tables():
    # T = 5*7 = 35 tokens per frame, 3 heads, 5 streams at different positions
    sh = W.Shape(batch=5, heads=3, chunk_frames=3, grid_h=5, grid_w=7, ring_frames=7)
    wl = W.Workload("ragged", sh, seed=11, history_starts=((),) * 5, measured_starts=(0, 3, 9, 30, 4),
                    window_frames=(7,))
    dev, ora = DevicePath(sh), OraclePath(sh)
    for rep in range(3):
        starts = [s + 3 * rep for s in wl.measured_starts]
        q, k, v = W.batch_qkv(wl, starts)
        q_out = dev.append(starts, q, k, v)
        q_ref = ora.append(starts, q, k, v)
        assert np.array_equal(to_bits(q_out), q_ref)
        assert_ring_equal(dev, ora)


def test_more_streams_than_one_launch_carries():
    sh = W.Shape(batch=37, heads=1, chunk_frames=1, grid_h=2, grid_w=3, ring_frames=4)
    wl = W.Workload("many", sh, seed=12, history_starts=((),) * 37,
                    measured_starts=tuple(range(37)), window_frames=(4,))
    dev, ora = DevicePath(sh), OraclePath(sh)
    q, k, v = W.batch_qkv(wl, wl.measured_starts)
    q_out = dev.append(wl.measured_starts, q, k, v)
    q_ref = ora.append(wl.measured_starts, q, k, v)
    assert np.array_equal(to_bits(q_out), q_ref)
    assert_ring_equal(dev, ora)


def test_library_table_feeds_append_bit_exact_where_tables_agree():
    # whole chain on the GPU with the library's own table: any ring difference must sit on a
    # table entry that differs from the oracle's (expected: none)
    wl = W.WORKLOADS["cfg1_wrapped"]
    dev, ora = DevicePath(wl.shape, use_oracle_table=False), OraclePath(wl.shape)
    stream_history(wl, dev, ora, check_ring=False)
    gk = to_bits(dev.ring_k)
    diff = gk != ora.ring.ring_k
    tables_equal = all(
        np.array_equal(dev.table(s)[0].cpu().numpy(), ora.table(s)[0]) and
        np.array_equal(dev.table(s)[1].cpu().numpy(), ora.table(s)[1]) for s in wl.history_starts[0])
    if tables_equal:
        assert not diff.any()
    else:
        assert diff.mean() < 1e-4
    assert np.array_equal(to_bits(dev.ring_v), ora.ring.ring_v)


@pytest.mark.parametrize("name", ["cfg2", "cfg5"])
def test_full_size_append_bit_exact(name):
    wl = W.WORKLOADS[name]
    dev, ora = DevicePath(wl.shape), OraclePath(wl.shape)
    s = wl.measured_starts
    q, k, v = W.batch_qkv(wl, s)
    q_out = dev.append(s, q, k, v)
    q_ref = ora.append(s, q, k, v)
    assert np.array_equal(to_bits(q_out), q_ref)
    assert_ring_equal(dev, ora)
