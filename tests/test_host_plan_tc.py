"""The chunk rule of the tensor-core inversion on the CPU (paper_1203_4587_gb300/csrc/host_logic.h):
at least one image column, never more scratch than 600 MB or a quarter more than the inverses it makes, and no less than
that allows."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_chunk_rule(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "check"
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_1203_4587_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host_plan_tc_check.cpp"), "-o", str(exe)], check=True,
                   capture_output=True, text=True, timeout=120)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout[-2000:]
