"""Launch rules of the kernels (plain C++ headers, compiled here with the host compiler)."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_13929_gb300", "csrc")
SOURCE = r"""
#include "spmc_plan.h"
extern "C" int pass_steps(int option, double mus, double porosity) { return spmc::pass_steps(option, mus, porosity); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rules")
    src, lib = d / "rules.cpp", d / "rules.so"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(lib), str(src)], check=True)
    r = ctypes.CDLL(str(lib))
    r.pass_steps.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_double]
    return r


@pytest.mark.parametrize("option", [1, 3, 8, 16, 29, 64])
@pytest.mark.parametrize("mus,porosity", [(0.5, 0.70), (2.0, 0.5), (0.5, 0.90), (0.0, 0.9), (0.3, 1.0)])
def test_a_pass_length_that_was_set_is_taken(rules, option, mus, porosity):
    assert rules.pass_steps(option, mus, porosity) == option


def test_automatic_pass_length_follows_the_optics(rules):
    assert rules.pass_steps(0, 0.5, 0.70) == 4          # an interaction every 10 steps
    assert rules.pass_steps(0, 0.5, 0.90) == 8          # every 30
    assert rules.pass_steps(0, 0.0, 0.5) == 8
