"""The FP32 work list's closed form on the CPU: tests/list_check.cu, built and run as
tests/plan_check.cu is."""
import os
import subprocess

import pytest

import paper_2603_02059_gb300 as tk
from test_plan_host import ROOT, _nvcc


def test_fp32_work_list_closed_form(tmp_path):
    tk.lib()
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    libdir = os.path.dirname(tk.LIB_PATH)
    exe = str(tmp_path / "list_check")
    cmd = [nvcc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-o", exe,
           os.path.join(ROOT, "tests", "list_check.cu"), "-L", libdir, "-ltraknn",
           "-Xlinker", "-rpath", "-Xlinker", libdir]
    build = subprocess.run(cmd, capture_output=True, text=True, timeout=600)
    assert build.returncode == 0, build.stderr[-3000:]
    run = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout[-3000:] + run.stderr[-2000:]
    assert "list check ok" in run.stdout
