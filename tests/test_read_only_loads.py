"""Kernels of a frame start while the one before them still runs, so the read-only
path (__ldg, ld.global.nc: data that nothing writes while the kernel lives) is only
for what no kernel of the chain writes.  Every such load of the chain's sources must
be one of these: theta, descriptors and maps, scene data, the caller's gradient.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_01074_gb300", "csrc")

READ_ONLY = [
    r"a\.theta\b",                                       # the caller's parameters
    r"a\.block_map \+ \w+(\.x)?$", r"row_map \+ g$",     # launch maps, uploaded with the plan
    r"sc\.mat_orig \+", r"(tp|p|q)( \+ [12])?$",         # scene data: materials, triangles
    r"reinterpret_cast<const float4\*>\(grad \+",        # the caller's gradient
    r"reinterpret_cast<const uint32_t\*>\(src\) \+ i$",  # copy_words: descriptors
]


def arguments(text, name):
    for m in re.finditer(re.escape(name) + r"\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text[m.end():i - 1]


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//.*", "", text)


def test_only_unwritten_data_goes_by_the_read_only_path():
    seen = 0
    for name in ("trace.cu", "render.cu", "sonar_internal.cuh"):
        for arg in arguments(source(name), "__ldg"):
            assert any(re.match(p, arg) for p in READ_ONLY), (name, arg)
            seen += 1
        assert "ld.global.nc" not in source(name)
    assert seen > 20
    # the nodes of a scene, by the two loads of devmath.cuh
    assert source("devmath.cuh").count("ld.global.nc") == 2
