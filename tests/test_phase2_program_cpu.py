"""The forward kernels' phase-2 program (phase2_program in csrc/tami_internal.h), on random product
tries: a C++ harness walks it as the kernels do and compares every group's factors with the trie's.
On the GPU the values of the two kernels that evaluate the trie in different ways are compared bit
for bit in test_gpu_small_launches.py."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_every_group_ends_on_its_product(tmp_path, seed):
    exe = str(tmp_path / "phase2_cases")
    cmd = ["g++", "-std=c++17", "-O1", "-D_GLIBCXX_ASSERTIONS", os.path.join(ROOT, "tests", "native", "phase2_cases.cpp"),
           "-I", os.path.join(ROOT, "paper_2311_17189_gb300", "csrc"), "-o", exe]
    subprocess.run(cmd, check=True, capture_output=True)
    r = subprocess.run([exe, str(seed)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
