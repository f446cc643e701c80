"""The series of e^x - 1 in the FP32 V-cycles (csrc/em1_series.h), compiled as host C++,
against long double.

The first omitted term is x^8/8!: (0.35)^7/8! = 1.6e-8 of x, 1.9e-8 of e^x - 1 at
x = -0.35 (where that is 0.84 x).  FP32: that and the last product's and sum's roundings,
2^-24 each, and what the inner ones leave of theirs."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_series_against_long_double(tmp_path):
    exe = str(tmp_path / "em1")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-Wall", "-o", exe,
                    os.path.join(ROOT, "tests", "em1_check.cpp")], check=True)
    w64, w32, lo, hi, zero = subprocess.run([exe], check=True, capture_output=True,
                                            text=True).stdout.split()
    assert float(w64) <= 1.9e-8 and max(float(lo), float(hi)) <= 1.9e-8
    assert float(w32) <= 1.9e-8 + 3.0 * 2.0 ** -24
    assert zero == "1"
