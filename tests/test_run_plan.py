"""Host logic of the resident step kernel's plan (no GPU): builds tests/native/run_plan_check.cpp
with the runtime's sources and runs it over channels, periodic and closed boxes, random porous
media and batches (see the C++ file)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1707_00198_gb300", "csrc")


def test_run_plan_covers_every_node_and_every_dependence(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "run_plan_check")
    cmd = [cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           os.path.join(ROOT, "tests", "native", "run_plan_check.cpp"), os.path.join(CSRC, "lbcg_geom.cpp"),
           os.path.join(CSRC, "lbcg_plan.cpp"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "ALL OK" in r.stdout, r.stdout + r.stderr
