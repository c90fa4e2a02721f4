"""CPU-only: what a kernel that may start before its predecessor has ended must keep to, read from its source.

Such a kernel waits (grid_dep_wait) before it touches global memory, and what it reads then may have been
written while it was already resident.  The read-only path (ld.global.nc: __ldg, or a const __restrict__ pointer
that the compiler turns into it) is only for memory that nobody writes during the kernel's life, and neither
the wait nor an asm memory clobber orders it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_22622_b200", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def source(name):
    """The file without its comments."""
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)


def kernels(text):
    """{name: body} of the __global__ functions of a file."""
    found = {}
    for m in re.finditer(r"__global__\s+void\b", text):
        start = text.index("{", m.end())
        depth, end = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
            if depth == 0:
                break
        found[re.findall(r"(\w+_kernel)\s*\(", text[m.start():start])[-1]] = text[start:end]
    return found


ALL = {name: (f, body) for f in FILES for name, body in kernels(source(f)).items()}
EARLY = sorted({k for f in FILES for call in re.findall(r"launch_(?:dependent|spread)\b[^;]*;", source(f)) for k in re.findall(r"\w+_kernel\b", call)})


def test_the_early_kernels_are_found():
    assert EARLY == sorted(["attn_sm100_kernel", "qkv_gemm_kernel", "qkv_finish_kernel", "bwd_delta_kernel", "bwd_kernel",
                            "rope_table_kernel", "rope_append_kernel", "rope_append_e4m3_kernel",
                            "norm_rope_append_kernel", "stage_e4m3_kernel"])
    assert set(EARLY) <= set(ALL)


@pytest.mark.parametrize("name", EARLY)
def test_an_early_kernel_waits_once(name):
    assert ALL[name][1].count("grid_dep_wait()") == 1 and ALL[name][1].count("grid_dep_launch()") == 1


@pytest.mark.parametrize("name", EARLY)
def test_nothing_is_read_before_the_wait(name):
    """Neither by a copy or a load that the kernel's own text shows, nor by a function that it calls with the launch's pointers."""
    before = ALL[name][1].split("grid_dep_wait()")[0]
    assert not re.search(r"tma_load\w*\(|bulk_\w+\(|__ld\w+\(|atomic\w+\(|\*>\(p\.status|\bp\.(q|k|v|x|out|d_out|lse|delta|counters|partial|[thw]_tab)\b", before)
    assert not re.search(r"\brun\(|load_tile\(|epilogue_rows[<(]|merge_\w+[<(]", before)


@pytest.mark.parametrize("name", sorted(set(ALL) - set(EARLY)))
def test_other_kernels_start_the_ordinary_way(name):
    assert "grid_dep" not in ALL[name][1]
    assert re.search(name + r"(<\w+>)?<<<", source(ALL[name][0]))


@pytest.mark.parametrize("name", FILES)
def test_no_read_only_loads(name):
    text = source(name)
    assert "__ldg(" not in text and "global.nc" not in text and "__restrict__" not in text


@pytest.mark.parametrize("name", ["attn_sm100_kernel", "qkv_gemm_kernel", "bwd_kernel", "norm_rope_append_kernel"])
def test_barriers_are_set_up_before_the_wait(name):
    body = ALL[name][1]
    assert re.search(r"\b(mbar_init|init_barriers)\(", body[:body.index("grid_dep_wait()")])
