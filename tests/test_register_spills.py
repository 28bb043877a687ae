"""Spills that `ptxas -v` reports for the kernels whose register budget is tight (a CTA more per SM, or 576 threads)."""
import os
import re
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2101_01321_b200" / "csrc"


def _spills(source, tmp_path):
    """{demangled kernel name: bytes of spill stores and loads}"""
    r = subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O3",
                        "-lineinfo", "-std=c++17", "--fmad=false", "-Xptxas", "-v", "-c", "-o", str(tmp_path / "o.o"), str(CSRC / source)],
                       check=True, capture_output=True, text=True)
    text = subprocess.run(["c++filt"], input=r.stderr, check=True, capture_output=True, text=True).stdout
    found = re.findall(r"Compiling entry function '[^']*?(\w+_kernel(?:<[^']*?>)?)\(.*?(\d+) bytes spill stores, (\d+) bytes spill loads", text, re.S)
    return {name: int(st) + int(ld) for name, st, ld in found}


@pytest.mark.parametrize("source,kernel,allowed", [("rowops.cu", "layernorm_pipe_kernel", 0), ("gemm_ln_i8.cu", "gemm_ln_kernel", 64)])
def test_spills(source, kernel, allowed, tmp_path):
    spills = {k: v for k, v in _spills(source, tmp_path).items() if k.startswith(kernel)}
    assert len(spills) > 3
    assert {k: v for k, v in spills.items() if v > allowed} == {}
