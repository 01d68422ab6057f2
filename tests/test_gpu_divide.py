"""The reciprocals and quotients of csrc/divide.cuh have the bits of the
device's division: every float of rcp_newton's range, and for the FP64
quotients random pairs, mantissas where rounding is hardest, and all
exponents (where div_by states no equality: the last place)."""
import subprocess
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu

HERE = Path(__file__).resolve().parent


def test_same_bits_as_the_division(tmp_path):
    from paper_2507_03975_gb300 import build
    exe = str(tmp_path / "divide_check")
    subprocess.check_call([build._nvcc(), *build.ARCH, "-std=c++17", "-O3", "-I" + build.CSRC,
                           str(HERE / "divide_check.cu"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
    lines = out.stdout.split("\n")[:-1]
    assert len(lines) >= 13 and all(line.split()[-1] == "0" for line in lines), out.stdout
