"""Host-side checks of the counting work-unit rule (no GPU), compiled from the library's own
header with the host C++ compiler."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2504_13445_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "native", "unit_rule_check.cpp")


def test_autotuner_and_batch_use_one_unit_size(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "unit_rule_check")
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-I", CSRC, SRC, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
