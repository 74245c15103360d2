"""Device code below the C ABI, checked by small programs built here with nvcc
against libgmls.so."""
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run(name, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2104_14447_gb300 import build

    lib = os.path.dirname(build.build())
    exe = str(tmp_path / name)
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.CSRC, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "device", name + ".cu"), "-L", lib, "-lgmls", "-Xlinker", "-rpath=" + lib,
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


def test_iterations_queued_past_the_end_write_nothing(tmp_path):
    assert "0 of 6" in _run("krylov_check", tmp_path)


def test_fp64_reciprocals(tmp_path):
    """The approximations are good to 2^-19 (20 mantissa bits read, 20 written), so
    the third-order steps leave 2^-57; what remains is rounding: half a unit of the
    last place of the result for the reciprocal, and for the root half of the
    rounding of x y in the step's residual (half a unit) besides."""
    root, reciprocal = (float(v) for v in _run("f64_math_check", tmp_path).split())
    assert root <= 1.5 and reciprocal <= 1.0
