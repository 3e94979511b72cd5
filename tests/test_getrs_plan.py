"""Host side of the solves with given factors: the block plans of
csrc/tl_getrs_plan.h over every n, number of right-hand sides and a range of
batches and shared-memory limits (cpu_helpers/getrs_plan_check.cpp).  Where no
block fits, tl_getrs_batched runs the register kernels instead."""
import os
import shutil
import subprocess
import tempfile

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_15217_gb300", "csrc")


def test_plans_fit_their_limits():
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "getrs_plan_check")
        subprocess.run([cxx, "-O2", "-std=c++17", "-I" + CSRC, os.path.join(HERE, "cpu_helpers", "getrs_plan_check.cpp"),
                        "-o", exe], check=True, capture_output=True)
        out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
