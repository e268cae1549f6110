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


def test_plans_of_lists_from_files(tmp_path):
    """A list read from a file whose operations are not the recursion's keeps them:
    no plan, made from the components' keys alone, stands in."""
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "list_file_check")
    src = os.path.join(ROOT, "tests", "host", "list_file_check.cpp")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fopenmp", "-I", os.path.join(ROOT, "include"), src, "-o", exe])
    res = subprocess.run([exe, str(tmp_path / "list.bin")], capture_output=True, text=True, timeout=600)
    assert res.returncode == 0 and res.stdout.strip().endswith("OK"), res.stdout + res.stderr


@pytest.mark.parametrize("spec,kind", [
    (dict(n_p=2, n_n=2, dirac_dim=2), "minors"), (dict(n_p=1, n_n=1, dirac_dim=2), "recursion"),
    (dict(n_p=2, n_n=2, dirac_dim=2, list_free=True), "recursion"),
    (dict(n_p=2, n_n=1, dirac_dim=4, spins=[((0, 1, 0), (0, 1, 0))]), "pair"),
])
def test_form_of_a_list(spec, kind):
    import paper_1301_4895_gb300 as mbc
    tl = mbc.build_term_list(**spec)
    assert tl.form()[0] == kind and tl.form()[1] > 0
    assert tl.form(mbc.SINK_BLOCK_MOMENTUM)[0] == ("recursion" if spec.get("list_free") else "pair")


def test_form_follows_the_precision():
    """A relativistic pn list fits the FP64 shared-memory kernel, but not the operation
    words of the mixed one: mixed calls take its pair form on the wave kernels."""
    import paper_1301_4895_gb300 as mbc
    tl = mbc.build_term_list(1, 1, 4, spins=[((0, 3), (1, 2))])
    assert tl.form(0, mbc.FP64)[0] == "recursion" and tl.form(0, mbc.MIXED)[0] == "pair"
    he3 = mbc.build_term_list(2, 1, 2)
    assert he3.form(0, mbc.FP64) == he3.form(0, mbc.MIXED)
