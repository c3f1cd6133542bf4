"""Parts of the work plan, checked by host programs: the closed form of a one-m-tile window's plan equals the general
search (tests/plan_single.cu), and the SIMT kernel's row groups hold over all sizes (tests/plan_simt.cu)."""

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(tmp_path, name, *flags):
    from paper_2609_33887_gb300 import build

    try:
        nvcc = build._nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    exe = str(tmp_path / name)
    subprocess.run([nvcc, "-std=c++17", *flags, "-I" + build.CSRC, "-o", exe,
                    os.path.join(ROOT, "tests", name + ".cu")], check=True, capture_output=True)
    return map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())


def test_closed_form_equals_the_search(tmp_path):
    n, differ = run(tmp_path, "plan_single")
    assert n > 100000 and differ == 0


def test_row_groups_of_the_simt_kernel(tmp_path):
    n, bad = run(tmp_path, "plan_simt", "-Xcompiler", "-fsanitize=signed-integer-overflow",
                 "-Xcompiler", "-fsanitize-undefined-trap-on-error")
    assert n > 5000 and bad == 0
