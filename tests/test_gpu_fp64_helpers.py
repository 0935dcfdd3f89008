"""The FP64 solver's reciprocal, root, halving, h^(-7/3), cut to FP32 and FP32 shock pre-test
against CUDA's own operations: tests/fp64_helpers_check.cu, compiled with the library's flags."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_helpers_keep_their_bounds(tmp_path):
    from paper_2010_02003_gb300 import build

    exe = tmp_path / "check"
    subprocess.check_call([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-prec-div=false",
                           "-prec-sqrt=false", "-ftz=true",
                           "-I", os.path.join(ROOT, "paper_2010_02003_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), "-o", str(exe),
                           os.path.join(ROOT, "tests", "fp64_helpers_check.cu")])
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    print(out.stdout)
    assert out.returncode == 0, out.stdout
