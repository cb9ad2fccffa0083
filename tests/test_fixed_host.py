"""The fixed-point sums of csrc/bits.cuh (host-compilable) against exact sums."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_sums_match_exact_sums(tmp_path):
    exe = tmp_path / "fixed_check"
    subprocess.run(["g++", "-std=c++17", "-O2", "-I",
                    os.path.join(ROOT, "paper_1906_01632_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fixed_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout
