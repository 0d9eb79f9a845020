"""bench.py's account of the arithmetic a launch runs in (no GPU)."""

import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_under_test", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


@pytest.mark.parametrize("kernel,precond,staged,want", [
    ("bicgstab_packed_kernel", 1, True, "int64"), ("cg_kernel", 1, True, "int64"), ("cg_kernel", 1, False, "fp64"),
    ("cg_packed_kernel", 0, True, "fp64"), ("gmres_kernel", 1, True, "fp64"), ("varteam_kernel", 1, True, "int64"),
    ("bicgstab_kernel", 1, False, "fp64"), ("bicgstab_ilu_packed_kernel", 2, True, "fp64")])
def test_arithmetic_follows_kernel_preconditioner_and_staging(bench, kernel, precond, staged, want):
    assert bench.arithmetic(kernel, precond, staged) == want
