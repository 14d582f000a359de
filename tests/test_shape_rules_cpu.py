"""CPU checks of host rules that pick kernel shapes (headers of csrc compiled with the host compiler)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host C++ compiler")
@pytest.mark.parametrize("name", ["sweep_shape", "factor_choice"])
def test_rule(name, tmp_path):
    exe = str(tmp_path / name)
    src = os.path.join(ROOT, "tests", "cpp", name + "_check.cpp")
    inc = os.path.join(ROOT, "paper_2301_10762_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-I", inc, src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
