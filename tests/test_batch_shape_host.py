"""Launch shapes of the batched solve (csrc/batch_shape.h): the tuner times the launch that
an untuned batch gets, and a tuned shape launches as the same shape untuned."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_shapes_over_amounts_of_work(tmp_path):
    exe = str(tmp_path / "shape")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-o", exe,
                    os.path.join(ROOT, "tests", "batch_shape_check.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["1"] * 6, out
