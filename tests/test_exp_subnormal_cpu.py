"""The kernels' exponential (csrc/tami_devmath.cuh) keeps values below the normal range, compiled for the
host against long double; so do the generated kernels whose products keep them."""
import os
import subprocess

import paper_2311_17189_gb300 as T
from paper_2311_17189_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2311_17189_gb300", "csrc", "tami_devmath.cuh")
ESTIMATE = 'asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));'


def test_exponential_below_the_normal_range(tmp_path):
    text = open(HEADER).read()
    assert text.count(ESTIMATE) == 1
    (tmp_path / "devmath_host.h").write_text(text.replace(ESTIMATE, "y = host_rcp_estimate(x);").replace("#pragma once", ""))
    exe = tmp_path / "cases"
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-w", "-I", str(tmp_path),
                    os.path.join(ROOT, "tests", "native", "exp_subnormal_cases.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-2000:]


def test_generated_kernels_that_keep_subnormal_values():
    """Every energy-input kernel and the Monte Carlo kernels of tables above 256 pole-DAG ops."""
    for order, code in ((4, W.ORDER4["code"]), (5, W.ORDER5["code"])):
        d = next(x for x in T.enumerate_sigma(order) if x["code"] == tuple(code))
        D = T.Diagram(d["alpha"], eps=d["eps"])
        for kind in ("fused", "forward", "adjoint", "energy"):
            keeps = kind == "energy" or D.info()["n_dag_ops"] > 256
            assert ("exp_neg<kFermiExp>" in D.jit_source(kind)) == keeps, (order, kind)
