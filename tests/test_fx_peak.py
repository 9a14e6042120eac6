"""The block fixed-point line FFT on lines that stand between its two scale
rules: a peak over a dense background, slow decay.  On the host, against long
double and the same passes in FP64, whose error it must not exceed
(tests/fx_peak_check.cu)."""

import os
import subprocess

import pytest

from test_fx_line import HERE, _nvcc


def test_fx_peak_host_check(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = tmp_path / "fx_peak_check"
    build = subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-x", "cu",
                            os.path.join(HERE, "fx_peak_check.cu"), "-o", str(exe)],
                           capture_output=True, text=True, timeout=600)
    assert build.returncode == 0, build.stderr
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout + run.stderr
    assert "OK" in run.stdout
