"""The 2-norm error of the fixed-point double transforms over that of the radix-4 passes in double, both
against long double, where test_host_fx does not compare them: single-mode inputs, and amplitudes that
put 9/8 of the sum of moduli anywhere between two powers of two (the unit is the coarser, the nearer to
the lower one it falls): never above 1."""
import shutil
import subprocess

import pytest

from paper_2007_06427_gb300 import build as B
from test_host_fx import PROG


@pytest.mark.parametrize("lg", range(3, 11))
def test_no_further_off_than_a_double_transform(lg, tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.getbasetemp()
    exe = d / "fx_ratio"
    if not exe.exists():
        (d / "fx_ratio.cpp").write_text(PROG)
        subprocess.run([cxx, "-std=c++17", "-O2", "-w", "-I", B.CSRC, str(d / "fx_ratio.cpp"), "-o", str(exe)], check=True)
    for mode in range(4):
        for amp in ("1", "0.9", "0.8", "0.72", "0.66", "0.6", "0.53"):
            out = subprocess.run([str(exe), str(lg), str(mode), amp], check=True, capture_output=True, text=True).stdout
            assert float(out.split()[1]) <= 1.0, (mode, amp)
