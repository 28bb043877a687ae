"""Spills and registers that `ptxas -v` reports for the kernels whose budget is tight (a CTA more per SM, or 576 threads)."""
import os
import re
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2101_01321_b200" / "csrc"


def _compiled(source, tmp_path):
    """{demangled kernel name: (bytes of spill stores and loads, registers)}"""
    r = subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O3",
                        "-lineinfo", "-std=c++17", "--fmad=false", "-Xptxas", "-v", "-c", "-o", str(tmp_path / "o.o"), str(CSRC / source)],
                       check=True, capture_output=True, text=True)
    text = subprocess.run(["c++filt"], input=r.stderr, check=True, capture_output=True, text=True).stdout
    found = re.findall(r"Compiling entry function '[^']*?(\w+_kernel(?:<[^']*?>)?)\(.*?(\d+) bytes spill stores, (\d+) bytes spill loads"
                       r".*?Used (\d+) registers", text, re.S)
    return {name: (int(st) + int(ld), int(regs)) for name, st, ld, regs in found}


@pytest.mark.parametrize("source,kernel,allowed", [("rowops.cu", "layernorm_pipe_kernel", 0), ("gemm_ln_i8.cu", "gemm_ln_kernel", 64)])
def test_spills(source, kernel, allowed, tmp_path):
    spills = {k: v[0] for k, v in _compiled(source, tmp_path).items() if k.startswith(kernel)}
    assert len(spills) > 3
    assert {k: v for k, v in spills.items() if v > allowed} == {}


def test_registers_of_the_light_one_wave_kernels(tmp_path):
    """512 threads: with more than 32 registers a short reduction has three CTAs per SM instead of four."""
    found = _compiled("gemm_small_i8.cu", tmp_path)
    light = {f"gemm_small_kernel<{kind}, true>": 32 for kind in (0, 1, 4, 5)}      # int8, Q16, h-GELU, Q16 as int16
    assert {k: found[k][1] for k in light if found[k][1] > light[k]} == {}
