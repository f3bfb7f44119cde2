"""Kernels that start before the kernel in front of them has ended (csrc/common.h, launch_overlapped) may
not read their inputs through loads that the compiler or the read-only cache may take from before their
grid_wait().  Nothing on a GPU shows such a load reliably, so the sources are looked at."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_32518_b200", "csrc")


def kernels(name):
    text = open(os.path.join(CSRC, name)).read()
    for m in re.finditer(r"__global__[^;{]*?(\w+_kernel)\(([^{;]*?)\)\s*\{", text, re.S):
        end = text.find("\n}\n", m.end())
        yield m.group(1), m.group(2), text[m.end():end]


@pytest.mark.parametrize("source", ["rope.cu", "attn.cu"])
def test_inputs_of_overlapped_kernels_are_read_behind_the_wait(source):
    found = [(name, params, body) for name, params, body in kernels(source) if "grid_wait()" in body]
    assert found
    for name, params, body in found:
        assert not re.search(r"const\s+(?!__grid_constant__)\w+\s*\*\s*__restrict__", params), name
        assert "__ldg(" not in body, name


def test_addresses_of_the_appends_take_the_wait_in():
    bodies = {name: body for name, _, body in kernels("rope.cu")}
    append = bodies["rope_kv_append_kernel"]
    assert re.search(r"in_idx = [^;]*\bbehind;", append) and re.search(r"tab = [^;]*\bbehind;", append, re.S)
    assert "lane = (threadIdx.x & 31) + grid_wait();" in bodies["rmsnorm_rope_kv_append_kernel"]
    assert "tid = threadIdx.x + grid_wait();" in bodies["rmsnorm_rope_kv_append_token_kernel"]
