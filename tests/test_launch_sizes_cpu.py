"""The table of shared-memory limits and resident blocks (csrc/tami_internal.h, LaunchSizes) on the host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_limits_never_fall(tmp_path):
    exe = str(tmp_path / "launch_sizes_cases")
    subprocess.run(["g++", "-std=c++17", "-O1", "-D_GLIBCXX_ASSERTIONS",
                    os.path.join(ROOT, "tests", "native", "launch_sizes_cases.cpp"),
                    "-I", os.path.join(ROOT, "paper_2311_17189_gb300", "csrc"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
