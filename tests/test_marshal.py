"""The native marshalling of the binding: only exactly well-formed calls take it, they do what the
general path does, and every other call still ends in the general path's error."""

import pytest
import torch

import paper_2609_32518_b200 as U
from paper_2609_32518_b200 import binding

SHAPE = dict(batch=2, heads=3, chunk_frames=2, grid_h=9, grid_w=16, ring_frames=5)
BF16 = torch.bfloat16


def buffers(device, sink=0, seed=0):
    sh = U.Shape.make(**SHAPE)
    gen = torch.Generator().manual_seed(seed)
    act = (sh.batch, sh.chunk_tokens, sh.heads, 128)
    cache = (sh.batch, sink + sh.ring_frames, sh.tokens_per_frame, sh.heads, 128)

    def normal(dims, dtype=BF16):
        return torch.randn(dims, generator=gen).to(dtype).to(device)

    return sh, {"q": normal(act), "k": normal(act), "v": normal(act), "q_out": normal(act), "out": normal(act),
                "ck": normal(cache), "cv": normal(cache), "cos": normal((sh.chunk_tokens, 64), torch.float32),
                "sin": normal((sh.chunk_tokens, 64), torch.float32), "gq": normal((sh.heads * 128,), torch.float32),
                "gk": normal((sh.heads * 128,), torch.float32)}


def calls(sh, t, sink):
    starts = [4, 6]
    app = (t["q"], t["k"], t["v"])
    tail = (t["cos"], t["sin"], t["q_out"], t["ck"], t["cv"])
    kv = (t["q"], t["ck"], t["cv"], t["out"])
    out = {
        "rmsnorm_rope_kv_append": (sh, sink, starts, *app, t["gq"], t["gk"], 1e-6, *tail, 0, None),
        "rope_kv_append_sink": (sh, sink, starts, *app, *tail, 0, None),
        "window_attn_sink": (sh, sink, starts, 4, min(sink, 1), *kv, None),
    }
    if sink == 0:
        out.update({
            "rope_table": (sh, 7, t["cos"], t["sin"], None),
            "rope_kv_append": (sh, starts, *app, *tail, 0, None),
            "window_attn": (sh, starts, 4, *kv, None),
            "window_attn_noalloc": (sh, starts, 4, *kv, None),
        })
    return out


def test_malformed_calls_end_in_the_general_path():
    sh, t = buffers("cpu")
    for name, args in calls(sh, t, 0).items():
        with pytest.raises(TypeError, match="expected a CUDA tensor"):
            getattr(U, name)(*args)
    with pytest.raises(ValueError, match="one entry per stream"):
        U.window_attn(sh, [1], 4, t["q"], t["ck"], t["cv"], t["out"])
    native = binding._native()
    assert native.rope_table(sh, 0, t["cos"], t["sin"]) is None              # argument missing
    assert native.rope_table(None, 0, t["cos"], t["sin"], None) is None      # not a Shape
    assert native.rope_table(sh, 1 << 40, t["cos"], t["sin"], None) is None  # not a 32-bit integer
    assert native.attn(sh, [1, 2], 4.0, t["q"], t["ck"], t["cv"], t["out"], None) is None


@pytest.mark.parametrize("broken", ["no compiler", "no nvcc", "module does not load"])
def test_calls_do_without_the_module(broken, monkeypatch, tmp_path):
    if broken == "module does not load":
        (tmp_path / "m.so").write_bytes(b"not a library")
        monkeypatch.setattr(binding._build, "build_marshal", lambda force=False: str(tmp_path / "m.so"))
    else:
        monkeypatch.setattr(binding._build, "marshal_path", lambda: str(tmp_path / "absent.so"))
        if broken == "no compiler":
            monkeypatch.setenv("CXX", str(tmp_path / "no-such-compiler"))
        else:
            def no_nvcc():
                raise RuntimeError("nvcc not found")
            monkeypatch.setattr(binding._build, "_nvcc", no_nvcc)
    binding.lib()
    monkeypatch.setattr(binding, "_fast", None)
    sh, t = buffers("cpu")
    with pytest.warns(RuntimeWarning, match="marshalled by ctypes"):
        with pytest.raises(TypeError, match="expected a CUDA tensor"):   # the general path's answer
            U.rope_table(sh, 7, t["cos"], t["sin"])
    for name, args in calls(sh, t, 0).items():                           # and no second warning
        with pytest.raises(TypeError, match="expected a CUDA tensor"):
            getattr(U, name)(*args)


def test_the_file_of_the_module_names_torch_and_python():
    import sysconfig
    path = binding._build.marshal_path()
    assert path.endswith(sysconfig.get_config_var("EXT_SUFFIX")) and torch.__version__.split("+")[0] in path


@pytest.mark.gpu
def test_well_formed_calls_take_the_module():
    for sink in (0, 2):
        sh, t = buffers("cuda", sink)
        native, made = binding._native(), calls(sh, t, sink)
        s, ap = made["rmsnorm_rope_kv_append"], made["rope_kv_append_sink"]
        assert native.norm_append(*s) == 0 and native.append(*ap) == 0 and native.attn_sink(*made["window_attn_sink"]) == 0
        if sink == 0:
            assert native.rope_table(*made["rope_table"]) == 0
            assert native.attn(*made["window_attn"]) == 0 and native.attn_noalloc(*made["window_attn_noalloc"]) == 0
    assert U.poll_status() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("sink", [0, 2])
def test_same_results_as_the_general_path(sink):
    for name in calls(*buffers("cpu", sink), sink):
        got, want = [], []
        for fn, results in ((getattr(U, name), got), (getattr(binding, "_general_" + name), want)):
            sh, t = buffers("cuda", sink)
            fn(*calls(sh, t, sink)[name])
            torch.cuda.synchronize()
            results += [t[n].cpu() for n in sorted(t)]
        for a, b in zip(got, want):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), name
    assert U.poll_status() == 0


@pytest.mark.gpu
def test_errors_on_cuda_tensors():
    sh, t = buffers("cuda")
    for bad in (t["q"].float(), t["q"][:1], t["q"].transpose(1, 2)):
        with pytest.raises(ValueError, match="q_rot: expected contiguous"):
            U.window_attn(sh, [4, 6], 4, bad, t["ck"], t["cv"], t["out"])
    with pytest.raises(U.UnstepError):
        U.window_attn(sh, [4, 6], 6, t["q"], t["ck"], t["cv"], t["out"])     # window longer than the ring
    with pytest.raises(U.UnstepError):
        U.rope_table(sh, -1, t["cos"], t["sin"])
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    U.rope_table(sh, 3, t["cos"], t["sin"], stream=side)
    side.synchronize()
    want = torch.empty_like(t["cos"])
    U.rope_table(sh, 3, want, t["sin"], stream=torch.cuda.current_stream().cuda_stream)
    assert torch.equal(t["cos"], want)
