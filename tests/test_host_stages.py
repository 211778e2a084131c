"""The stage radices of the FFTs on the CPU, over every length from 1 to 1024
(paper_1203_4587_gb300/csrc/host_logic.h: fft_stages), and that the check notices a slip."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1203_4587_gb300", "csrc")


def run(tmp_path, inc):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "check"
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-I", str(inc), os.path.join(ROOT, "tests", "host_stages_check.cpp"),
                    "-o", str(exe)], check=True, capture_output=True, text=True, timeout=120)
    return subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)


def test_stages(tmp_path):
    r = run(tmp_path, CSRC)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout[-2000:]


@pytest.mark.parametrize("old,new", [("two == 4 || two == 2 ? 2 :", "two == 4 ? 2 :"), ("two == 1 ? 1 : 3", "3"),
                                     ("for (int k = nf - 1; k >= 0; --k) {\n    if (f[k] == 4) two += 2;", "for (int k = nf - 1; k >= 0; --k) {\n    if (f[k] == 4) two += 1;")])
def test_check_notices_a_slip(tmp_path, old, new):
    src = open(os.path.join(CSRC, "host_logic.h")).read()
    assert src.count(old) == 1
    (tmp_path / "host_logic.h").write_text(src.replace(old, new))
    r = run(tmp_path, tmp_path)
    assert r.returncode != 0 and "FAIL" in r.stdout
