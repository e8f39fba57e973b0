"""The quantizer's three-bit codes by rank of the coefficients, on the CPU, against the sorted table (three_bit_levels.cpp)."""
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_three_bit_codes_equal_those_of_the_sorted_table(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    exe = str(tmp_path / "levels")
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", include, "-I", os.path.join(ROOT, "paper_1802_00150_b200", "csrc"),
                        os.path.join(HERE, "three_bit_levels.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
