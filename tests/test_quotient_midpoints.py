"""The refined quotient is correctly rounded: near the middle of two binary32
numbers, where alone it could fail, by enumeration."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_quotients_next_to_a_midpoint(tmp_path):
    if shutil.which("gcc") is None:
        pytest.skip("gcc not available")
    exe = str(tmp_path / "midpoints")
    subprocess.run(["gcc", "-O2", "-std=c11", "-ffp-contract=off", os.path.join(HERE, "quotient_midpoints.c"), "-o", exe,
                    "-lm"], check=True)
    cases, wrong = (int(v) for v in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split())
    assert cases == 69778209 and wrong == 0
