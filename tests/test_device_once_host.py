"""Settings that belong to a device (csrc/device_once.h): made on every device that a
process uses, and none of the launchers keeps them per process."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1305_2418_gb300", "csrc")


def test_once_per_device(tmp_path):
    exe = str(tmp_path / "once")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-o", exe,
                    os.path.join(ROOT, "tests", "device_once_check.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["1"] * 4, out


def test_no_launcher_remembers_an_attribute_per_process():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            assert not re.search(r"static\s+bool\s+\w+\s*=", f.read()), name
