"""The windows' index arithmetic modulo 2^32 on the host, built so that signed
overflow traps: the library's device header, every window shape, origins from
0 to the largest lattice index."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_index_arithmetic_stays_unsigned(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "index_check"
    subprocess.check_call([cxx, "-O1", "-std=c++17", "-fsanitize=signed-integer-overflow",
                           "-fsanitize-undefined-trap-on-error",
                           "-include", "math.h", "-I", os.path.join(ROOT, "paper_2501_12581_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "index_check.cpp"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    assert int(out) == 5 * 6 ** 3 * 512
