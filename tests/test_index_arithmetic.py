"""The kernels' index arithmetic (csrc/pf_index.h) on the CPU, at shapes where a mistake
would read or write out of range: index_arithmetic.cpp runs the functions the kernels call."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1202_6163_gb300", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    out = str(tmp_path_factory.mktemp("index") / "index_arithmetic")
    subprocess.run([gxx, "-O1", "-std=c++17", "-Wall", "-Werror", "-ftrapv", "-I", CSRC, "-o", out,
                    os.path.join(HERE, "index_arithmetic.cpp")], check=True)
    return out


@pytest.mark.parametrize("what", ["strata", "permute_parts", "runs_and_chunks", "rows"])
def test_index_arithmetic(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
