"""The closed form of a one-m-tile window's plan equals the general search (tests/plan_single.cu, a host program)."""

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_closed_form_equals_the_search(tmp_path):
    from paper_2609_33887_gb300 import build

    try:
        nvcc = build._nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    exe = str(tmp_path / "plan_single")
    subprocess.run([nvcc, "-std=c++17", "-I" + build.CSRC, "-o", exe, os.path.join(ROOT, "tests", "plan_single.cu")],
                   check=True, capture_output=True)
    n, differ = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert n > 100000 and differ == 0
