"""The kernels' sine (csrc/tami_devmath.cuh) keeps its relative accuracy next to its zeros, compiled for
the host against long double."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2311_17189_gb300", "csrc", "tami_devmath.cuh")
ESTIMATE = 'asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));'


def test_sine_next_to_its_zeros(tmp_path):
    text = open(HEADER).read()
    assert text.count(ESTIMATE) == 1
    (tmp_path / "devmath_host.h").write_text(text.replace(ESTIMATE, "y = host_rcp_estimate(x);").replace("#pragma once", ""))
    exe = tmp_path / "cases"
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-w", "-I", str(tmp_path),
                    os.path.join(ROOT, "tests", "native", "trig_zero_cases.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-2000:]
