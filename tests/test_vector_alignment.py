"""The channel vectors of the surrogate's data-moving kernels are moved with
16-byte accesses, so they have to be aligned for them wherever the compiler
keeps them: an array of 2-byte elements that stays in local memory (a debug
build, a spill) may otherwise start off a 16-byte boundary.  Checked by the
compiler, no GPU needed."""
import os
import subprocess

import pytest

from paper_1711_03254_gb300 import build

CHECK = """
#include "{src}"
static_assert(alignof(ws::Vec<8>) == 16 && sizeof(ws::Vec<8>) == 16, "8 BF16 values move as one 16-byte access");
static_assert(alignof(ws::Vec<1>) == 2 && sizeof(ws::Vec<1>) == 2, "a scalar has the type's alignment");
static_assert(alignof(ws::Vec<8, float>) == 16 && sizeof(ws::Vec<8, float>) == 32, "8 FP32 values move as two");
static_assert(alignof(ws::Vec<1, float>) == 4 && sizeof(ws::Vec<1, float>) == 4, "a scalar has the type's alignment");
"""


def test_channel_vectors_are_aligned_for_their_accesses(tmp_path):
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src = tmp_path / "check.cu"
    src.write_text(CHECK.format(src=os.path.join(build.CSRC, "ws_ops.cu")))
    r = subprocess.run([cc, *build.ARCH, "-std=c++17", "--cuda", str(src), "-o", str(tmp_path / "check.ii")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
