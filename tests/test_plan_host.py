"""The evaluation plans (host code) give the components of the list's own
recursion on random propagators, with every operand index in range."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT


def test_plans_match_the_recursion(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "plan_check")
    src = os.path.join(ROOT, "tests", "host", "plan_check.cpp")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fopenmp", "-I", os.path.join(ROOT, "include"), src, "-o", exe])
    res = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert res.returncode == 0 and res.stdout.strip().endswith("OK"), res.stdout + res.stderr
