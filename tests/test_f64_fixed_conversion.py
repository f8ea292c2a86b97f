"""The integer-pipe conversion of the fixed-point node update (lbm_f64fx.cuh, from_fixed_int)
against the rounding conversion it stands in for, bit for bit, on the host."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("seed", [1, 2])
def test_integer_conversion_has_the_bits_of_the_rounding_conversion(tmp_path, seed):
    exe = str(tmp_path / "fxconv_check")
    r = subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-o", exe,
                        os.path.join(HERE, "native", "fxconv_check.cpp")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe, "300000", str(seed)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("0 failures"), r.stdout
