"""The constants of operator calls, without a GPU: operator_consts.cpp and host_consts.cpp linked with a host program that
stands in for the device side (operator_consts_host.cpp)."""
import os
import subprocess
from pathlib import Path

import pytest

HERE = Path(__file__).resolve().parent
CSRC = HERE.parent / "paper_2101_01321_b200" / "csrc"
CUDA = Path(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")).parent.parent


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = tmp_path_factory.mktemp("operator_consts") / "check"
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", f"-I{CSRC}", f"-I{CUDA / 'include'}", "-o", str(exe),
                    str(HERE / "operator_consts_host.cpp"), str(CSRC / "operator_consts.cpp"), str(CSRC / "host_consts.cpp")],
                   check=True)
    return str(exe)


@pytest.mark.parametrize("check", ["residual_search", "one_off", "in_use", "linear_keys"])
def test_operator_constants(program, check):
    r = subprocess.run([program, check], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
