"""The projector's Jacobi sweeps give the same bits in every kernel a rank may run in (alone: 32 or 128 threads up to
rank 16; in a grouped launch: 256), also where the decision for another sweep is a matter of the last bit, so that a
grouped solve equals a solo one.  Compiles tests/gpu_jacobi_check.cu and runs it."""
import os
import shutil
import subprocess

import pytest

from paper_1503_03004_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_jacobi_sweeps_do_not_depend_on_the_thread_count(tmp_path):
    nvcc = os.environ.get("NVCC", "nvcc")
    if shutil.which(nvcc) is None or not torch.cuda.is_available():
        pytest.skip("needs nvcc and a GPU")
    libdir = os.path.dirname(binding.LIB_PATH)
    exe = str(tmp_path / "gpu_jacobi_check")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                        "-o", exe, os.path.join(ROOT, "tests", "gpu_jacobi_check.cu"), "-L" + libdir, "-lsfr",
                        "-Xlinker", "-rpath=" + libdir], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-3000:]
