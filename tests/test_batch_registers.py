"""Registers of the batched temporal kernels.  With per-stream parameters (read through a run-time
index into registers) the FP32 form wants more than the 64 registers of four blocks a SM: with 152
bytes of spills a thread it was 3 % slower than with none, so it is compiled for three blocks."""
import re
import subprocess

import pytest

from paper_2312_06827_gb300 import _build

SOURCE = """
#include "svgf_batch.cuh"
template __global__ void svgf::batch::kb_temporal<svgf::dev::%s, %s>(const __grid_constant__ svgf::BatchTemporalArgs);
"""


def spill_stores(tmp_path, storage, uniform):
    try:
        nvcc = _build.nvcc_path()
    except RuntimeError:
        pytest.skip("no nvcc")
    src = tmp_path / "one.cu"
    src.write_text(SOURCE % (storage, uniform))
    r = subprocess.run([nvcc, *_build.NVCC_ARCH, "-O3", "-std=c++17", f"-I{_build.INCLUDE}", f"-I{_build.CSRC}", "-Xptxas", "-v",
                        "-c", str(src), "-o", str(tmp_path / "one.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    m = re.findall(r"Compiling entry function '\w*kb_temporal.*?(\d+) bytes spill stores", r.stderr, re.S)
    assert len(m) == 1, r.stderr
    return int(m[0])


def test_per_stream_fp32_form_spills_little(tmp_path):
    # 60 bytes with three blocks' 80 registers, 152 with four blocks' 64
    assert spill_stores(tmp_path, "StoreF32", "false") <= 80
