"""The integer division of the pair step (div_int, csrc/fp64_math.cuh), built
for the host, returns the division operator's bits: it is correctly rounded
by construction, so no tolerance. The reciprocal seed of the device is an
approximation (at most 2 units of its last place off), so the same holds with
the host's seed moved by that much and more."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("seed_ulp", [0, -2, 2, -4, 4])
def test_div_int_is_the_correctly_rounded_quotient(tmp_path, seed_ulp):
    exe = str(tmp_path / "div_int_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", f"-DSVM_DIV_SEED_ULP=({seed_ulp})",
                    "-I", os.path.join(ROOT, "paper_1406_5161_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "div_int_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe, "4000000"], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout
