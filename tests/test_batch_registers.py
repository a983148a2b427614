"""Registers of the batched temporal kernels: four blocks a SM leave a thread 64, and the descriptor of
the tile's stream (read through a run-time index into registers) has to fit beside the stage's own.
Kept over a walk of several tiles it did not: 152 bytes of spills a thread with per-stream parameters in
FP32, which was slower than the kernel before it."""
import re
import subprocess

import pytest

from paper_2312_06827_gb300 import _build

SOURCE = """
#include "svgf_batch.cuh"
template __global__ void svgf::batch::kb_temporal<svgf::dev::%s, %s>(const __grid_constant__ svgf::BatchTemporalArgs);
"""


@pytest.mark.parametrize("uniform", ["false", "true"])
@pytest.mark.parametrize("storage", ["StoreF32", "Store16<false>", "Store16<true>"])
def test_forms_spill_at_most_24_registers(tmp_path, storage, uniform):
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
    assert int(m[0]) <= 24 * 4
