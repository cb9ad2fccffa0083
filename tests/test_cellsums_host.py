"""The residual's cell sums (csrc/cellsums.cuh, host-compilable) against exact ones:
no less accurate than the FP64 form."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_cell_sums_are_no_less_accurate_than_fp64(tmp_path):
    exe = tmp_path / "cellsums_check"
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1906_01632_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "cellsums_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    print(r.stdout)
    assert r.returncode == 0, r.stdout
