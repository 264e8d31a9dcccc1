"""The kernels' fixed-point elementary functions (csrc/tami_devmath.cuh) on the host, compiled with
g++ behind stand-ins for CUDA's intrinsics, against long double."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2311_17189_gb300", "csrc", "tami_devmath.cuh")
ESTIMATE = 'asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));'


@pytest.fixture(scope="module")
def cases(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed_math")
    text = open(HEADER).read()
    assert text.count(ESTIMATE) == 1
    (d / "devmath_host.h").write_text(text.replace(ESTIMATE, "y = host_rcp_estimate(x);").replace("#pragma once", ""))
    exe = d / "cases"
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-w", "-I", str(d),
                    os.path.join(ROOT, "tests", "native", "fixed_math_cases.cpp"), "-o", str(exe)], check=True)
    return exe


@pytest.mark.parametrize("what", ["rcp", "exp", "trig"])
def test_fixed_point_function(cases, what):
    """Within 0.502 ulp (reciprocal), 0.51 ulp (e^t), 0.75 ulp (e^t - 1), 8e-17 absolute (cos, sin)."""
    r = subprocess.run([str(cases), what], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-2000:]
