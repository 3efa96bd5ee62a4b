"""Pinned rasters that a kernel reads through their device mapping: only where
the whole batch lies in one pinned range (checked on the CPU, no GPU involved)."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2104_14667_gb300", "csrc")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_range_check_at_its_edges(tmp_path):
    exe = tmp_path / "pinned_range_check"
    subprocess.run(["g++", "-std=c++17", "-O2", "-x", "c++", "-I", CSRC,
                    os.path.join(ROOT, "tests", "pinned_range_check.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and "failures 0" in out.stdout, out.stdout + out.stderr


def test_uploads_hand_a_kernel_checked_ranges_only():
    with open(os.path.join(CSRC, "api.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    start = text.index("int upload(composite_ctx")
    upload = text[start:text.index("\n}\n", start)]
    # the kernel's host rasters come from mapped_range over every byte that it may read
    assert "launch_repitch" in upload and "cudaHostGetDevicePointer" not in upload
    assert re.search(r"mapped_range\(src, \(c - 1\) \* stride \+ \(h - 1\) \* pitch \+ row\)", upload)
    start = text.index("const void *mapped_range(")
    assert "in_one_range" in text[start:text.index("\n}\n", start)]
