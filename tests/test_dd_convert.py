"""The set-up's integer split of a double into a float pair (csrc/rb_dd.cuh), built
for the host: the bits of the compiler's conversions for
every exponent, ties, both signs, zeros, subnormals, infinities and NaN."""
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent


@pytest.mark.parametrize("opt", ["-O0", "-O2"])
def test_integer_conversions_give_the_same_bits(tmp_path, opt):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "convert_check"
    subprocess.run([gxx, opt, "-std=c++17", "-ffp-contract=off", f"-I{ROOT / 'paper_2404_11397_gb300' / 'csrc'}",
                    str(ROOT / "tests" / "dd_host" / "convert_check.cpp"), "-o", str(exe)], check=True, capture_output=True)
    n, bad = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert n > 900000 and bad == 0
