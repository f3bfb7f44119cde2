"""Launches that overlap the kernel before them: a stream of dependent calls gives what the same calls
give with a synchronisation after each one, eagerly, on several streams and under capture."""

import pytest
import torch

import paper_2609_32518_b200 as U
from splits import forms, split_on_device

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16


class Layer:
    """One layer whose calls depend on one another: q_rot feeds the next chunk's q."""

    def __init__(self, seed, heads=3, norm=False, noalloc=False):
        self.sh = U.Shape.make(batch=1, heads=heads, chunk_frames=2, grid_h=9, grid_w=16, ring_frames=6)
        gen = torch.Generator().manual_seed(seed)
        act = (1, self.sh.chunk_tokens, heads, 128)
        cache = (1, 6, self.sh.tokens_per_frame, heads, 128)
        self.q, self.k, self.v = (torch.randn(act, generator=gen).to(BF16).cuda() for _ in range(3))
        self.ck, self.cv = (torch.randn(cache, generator=gen).to(BF16).cuda() for _ in range(2))
        self.gain = torch.rand(heads * 128, generator=gen).cuda()
        self.cos, self.sin = (torch.zeros(self.sh.chunk_tokens, 64, device="cuda") for _ in range(2))
        self.q_rot, self.out = torch.zeros_like(self.q), torch.zeros_like(self.q)
        self.norm, self.attn = norm, U.window_attn_noalloc if noalloc else U.window_attn
        # 77 heads and more are 154 items and more: a whole round, and parts merged through scratch behind it
        assert ("scratch" in forms(split_on_device(self.sh, [6], 6))) == (heads >= 77)

    def steps(self):
        # every call reads what the one before it wrote, and writes what the one before that read
        for start in range(6, 18, 2):
            yield lambda: U.rope_table(self.sh, start, self.cos, self.sin)
            if self.norm:
                yield lambda: U.rmsnorm_rope_kv_append(self.sh, 0, [start], self.q, self.k, self.v, self.gain, self.gain,
                                                       1e-6, self.cos, self.sin, self.q_rot, self.ck, self.cv)
            else:
                yield lambda: U.rope_kv_append(self.sh, [start], self.q, self.k, self.v, self.cos, self.sin, self.q_rot,
                                               self.ck, self.cv)
            yield lambda: self.attn(self.sh, [start], 6, self.q_rot, self.ck, self.cv, self.out)
            yield lambda: U.rope_kv_append(self.sh, [start], self.out, self.q_rot, self.v, self.cos, self.sin, self.q,
                                           self.ck, self.cv)

    def run(self, sync=False):
        for step in self.steps():
            step()
            if sync:
                torch.cuda.synchronize()

    def state(self):
        return [t.clone() for t in (self.q, self.q_rot, self.ck, self.cv, self.out, self.cos, self.sin)]


def same(a, b):
    return all(torch.equal(x.view(torch.uint8), y.view(torch.uint8)) for x, y in zip(a, b))


@pytest.mark.parametrize("norm,heads", [(False, 3), (True, 3), (False, 80)])
@pytest.mark.parametrize("noalloc", [False, True])
def test_dependent_calls_back_to_back(norm, noalloc, heads):
    want = Layer(1, heads, norm=norm, noalloc=noalloc)
    for _ in range(3):
        want.run(sync=True)
    for _ in range(4):
        got = Layer(1, heads, norm=norm, noalloc=noalloc)
        torch.cuda.synchronize()
        for _ in range(3):
            got.run()
        torch.cuda.synchronize()
        assert same(got.state(), want.state())
    assert U.poll_status() == 0


@pytest.mark.parametrize("heads", [(3, 12), (77, 80)])   # clusters, and parts in the scratch of either stream
def test_two_streams_at_once(heads):
    want = [Layer(s, heads=h) for s, h in zip((2, 3), heads)]
    got = [Layer(s, heads=h) for s, h in zip((2, 3), heads)]
    for layer in want:
        layer.run(sync=True)
    torch.cuda.synchronize()
    for layer in got:
        with torch.cuda.stream(torch.cuda.Stream()):
            layer.run()
    torch.cuda.synchronize()
    for g, w in zip(got, want):
        assert same(g.state(), w.state())


@pytest.mark.parametrize("noalloc,heads", [(False, 3), (True, 3), (False, 77), (True, 77)])
def test_under_capture_with_a_fork_and_a_join(noalloc, heads):
    want, got = Layer(4, heads, noalloc=noalloc), Layer(4, heads, noalloc=noalloc)
    other_want, other = Layer(5, heads), Layer(5, heads)
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    for stream, layer in ((main, Layer(6, heads, noalloc=noalloc)), (side, Layer(7, heads))):   # scratch of both streams
        with torch.cuda.stream(stream):
            layer.run()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        side.wait_stream(main)
        with torch.cuda.stream(side):
            other.run()
        got.run()
        main.wait_stream(side)
        U.rope_kv_append(got.sh, [2], other.q, other.k, other.v, got.cos, got.sin, got.q_rot, got.ck, got.cv)
    for _ in range(2):
        graph.replay()
        want.run(sync=True)
        other_want.run(sync=True)
        U.rope_kv_append(want.sh, [2], other_want.q, other_want.k, other_want.v, want.cos, want.sin, want.q_rot,
                         want.ck, want.cv)
    torch.cuda.synchronize()
    assert same(got.state(), want.state()) and same(other.state(), other_want.state())
    assert U.poll_status() == 0
