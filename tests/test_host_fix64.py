"""The fixed-point products of the float64 path (csrc/fix64.cuh) on the host: conversion, ranges, overflow at
the longest sum, and the error of a sum against the exact one and against the float64 loop it replaces.
Compiles tests/host_fix64_check.cu and runs it."""
import os
import platform
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_products(tmp_path):
    nvcc = os.environ.get("NVCC", "nvcc")
    if shutil.which(nvcc) is None:
        pytest.skip("nvcc not found")
    if platform.machine() != "x86_64":
        pytest.skip("the check's exact sums need 80-bit long doubles")
    exe = str(tmp_path / "host_fix64_check")
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-o", exe, os.path.join(ROOT, "tests", "host_fix64_check.cu")],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-3000:]
