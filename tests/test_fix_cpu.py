"""The fixed-point arithmetic of the FP64 transforms (csrc/fix_fft.h), compiled for the host and
checked against long double.  Bounds in units of the last place: sums are exact (long double
adds its own 2^-64 of 2^62); a product rounds twice and leaves out a product of two half-unit
words (3/4 a component, two components); dft3 halves two components and dft5 rounds four products
a component, dft8 one; shifts and conversions round once; ties to even leave no bias (its random
part over 10^5 draws is 0.35 / 316)."""
import pathlib
import shutil
import subprocess

import pytest

ROOT = pathlib.Path(__file__).resolve().parent.parent
BOUNDS = {"dft2": 0.5, "dft3": 2.5, "dft4": 1.0, "dft5": 3.0, "dft8": 2.0, "mul": 1.5, "conj": 1.5, "const": 1.0,
          "from": 0.5, "to": 0.0, "shift": 0.5, "bias": 0.005}


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_fixed_point_error_bounds(tmp_path):
    exe = tmp_path / "fix_check"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", str(ROOT / "paper_2512_04447_gb300" / "csrc"),
                    str(ROOT / "tests" / "native" / "fix_check.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    worst = {k: float(v) for k, v in (line.split() for line in out.strip().splitlines())}
    assert set(worst) == set(BOUNDS)
    for k, b in BOUNDS.items():
        assert worst[k] <= b, (k, worst[k])
