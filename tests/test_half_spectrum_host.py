"""The half-spectrum convolution's index rules (bte_internal.h), compiled for the
host: the sums over the stored pencils with their pair weights against the plain
sum over every mode after the real part of the inverse transform, and the visit
order of every tile. Tolerance: FP64 sums of up to 12^3 terms, 1e-12."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_half_spectrum_sums_match_the_plain_sum(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "half_spectrum_check"
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-o", str(exe),
                    os.path.join(HERE, "host", "half_spectrum_check.cu")], check=True, capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout.split("\n")
    rows = [r.split() for r in out if r.strip()]
    assert len(rows) == 8
    for kind, n, value in rows:
        assert float(value) <= (1e-12 if kind == "sum" else 0), (kind, n, value)
