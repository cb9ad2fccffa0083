"""bench.launch_model_bytes: the byte model of the kernels that run (the formulas of
elder_profile_read in include/elder.h)."""
import argparse

import pytest

import bench

CPN = 64 * 64 * 16 / (65 * 65 * 17)


@pytest.mark.parametrize("precision,smoother,cls,expected", [
    ("mixed", "zline", "smooth0", 16 * 4 + 1),
    ("fp64", "zline", "smooth0", 16 * 8 + 1),
    ("mixed", "jacobi", "smooth0", 8 * 4 + 1),
    ("mixed", "zline", "spmv", 8 * 4 + 2 * 4 * CPN + 1),
    ("mixed", "zline", "mg_residual", 8 * 4 + 2 * 4 * CPN + 1),
    ("mixed", "zline", "jacobian", 40 * 4 + 18 + 2 * 4 * CPN),
    ("mixed", "zline", "smooth", 26 * 4 + 2 * 4 * CPN + 2),
    ("mixed", "ilu", "spmv", 108 * 4 + 6 * 4 + 1),
    ("mixed", "ilu", "mg_residual", 108 * 2 + 6 * 4 + 1),
    ("fp64", "zline", "spmv", 108 * 8 + 6 * 8 + 1),
    ("mixed", "zline", "residual", 49 + 16 * CPN),
])
def test_bytes_per_node(precision, smoother, cls, expected):
    a = argparse.Namespace(precision=precision, smoother=smoother, grid=[64, 64, 16])
    assert bench.launch_model_bytes(a, cls) == pytest.approx(expected, rel=1e-12)
