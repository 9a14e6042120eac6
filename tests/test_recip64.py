"""The FP64 reciprocal psd::recip_pos (hardware estimate plus one third-order
step) against the IEEE quotient on the GPU: within 1 ulp over all positive doubles
tried, special values equal (tests/recip64_check.cu)."""

import os
import subprocess

import pytest

from test_recip import HERE, _nvcc

pytestmark = pytest.mark.gpu


def test_recip_pos_f64_within_one_ulp(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = tmp_path / "recip64_check"
    build = subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                            os.path.join(HERE, "recip64_check.cu"), "-o", str(exe)],
                           capture_output=True, text=True, timeout=600)
    assert build.returncode == 0, build.stderr
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert run.returncode == 0, run.stdout + run.stderr
    assert "OK" in run.stdout
