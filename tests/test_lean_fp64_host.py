"""The FP64 exponential and inverse square root with few FP64 instructions
(csrc/lean_fp64.cuh), compiled as host C++, against long double.

Bounds: one rounding of the table entry, of its product sum and of the reduced
argument (e^x below 1 ulp); two roundings and the estimate's product
(1/sqrt below 1.5 ulp)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_lean_functions_against_long_double(tmp_path):
    exe = str(tmp_path / "lean")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-o", exe,
                    os.path.join(ROOT, "tests", "lean_fp64_check.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert float(out[0]) <= 1.0 and float(out[1]) <= 1.5, out
    assert out[2:] == ["1", "1", "1"], out
