"""The register FFT (fft_reg.cuh) as the transforms of the FP64 operator (N = 8 .. 32) and of
N = 48 in FP32 use it, compiled for the host, against the dense sums; and the symmetry to the last bit
that the FP32 forward transforms of N = 8 and 16 rely on. Tolerance, as for FP32 at the smaller N:
about four units in the last place of the largest output (5e-7, 1e-15)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_register_fft_in_64_bits_and_at_n48(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "fft_wide_check"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-o", str(exe), os.path.join(HERE, "host", "fft_wide_check.cu")],
                   check=True, capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split("\n")
    rows = [r.split() for r in out if r.strip()]
    assert len(rows) == 26
    for r in rows:
        assert float(r[-1]) <= (0 if r[1] == "symmetry" else 1e-15 if r[1] == "f64" else 5e-7), r
