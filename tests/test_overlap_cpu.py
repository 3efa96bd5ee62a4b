"""Kernels launched while their predecessor drains, checked in the sources:
each of them waits for the stream's earlier work in every thread, before any
way out of the kernel and before its first use of a pointer into global memory."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_14667_gb300", "csrc")


def sources() -> dict:
    out = {}
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, name)) as f:
                out[name] = re.sub(r"//[^\n]*", "", f.read())
    return out


def overlapped_kernels() -> list:
    names = set()
    for text in sources().values():
        names |= set(re.findall(r"launch_overlapped\(\s*(\w+)", text))
    return sorted(names - {"void"})   # its own definition


def braces(text: str, start: int) -> str:
    depth = 0
    for i in range(text.index("{", start), len(text)):
        depth += (text[i] == "{") - (text[i] == "}")
        if depth == 0:
            return text[text.index("{", start) + 1:i]
    raise AssertionError("unbalanced braces")


def body_of(kernel: str) -> str:
    for text in sources().values():
        m = re.search(r"__global__[^;{]*\b" + kernel + r"\s*\(", text)
        if m:
            return braces(text, m.end())
    raise AssertionError(f"no definition of {kernel}")


def test_the_composite_path_is_covered():
    assert {"clear_plane_kernel", "count_linear_kernel", "depth_linear_kernel", "count_bits_kernel", "count_tma_kernel",
            "depth_tma_kernel", "count_bits_bulk_kernel", "render_counts_kernel",
            "render_mean_kernel"} <= set(overlapped_kernels())


@pytest.mark.parametrize("kernel", overlapped_kernels())
def test_waits_before_it_touches_memory(kernel):
    body = body_of(kernel)
    assert body.count("await_previous();") == 1
    before = body[:body.index("await_previous();")]
    assert "return" not in before
    # unconditional: at the outermost level of the kernel
    assert before.count("{") == before.count("}")
    # loads, stores and atomics of the kernels go through these
    for use in ("flags[", "flag_set", "plane[", "data[", "__ldcs", "__ldg", "atomic", "fold_", "load_unit", "safe_members",
                "tma_load", "bulk_load", "produce"):
        assert use not in before, use
