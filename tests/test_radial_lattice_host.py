"""The weights' closed forms on the grid's lattice (csrc/radial.h, Lattice), compiled for the host, against
the same forms in long double. Each is a handful of rounded operations with its phase reduced exactly, so
the error is within 12 units of 2^-53 of the terms that are subtracted, however large the phase; and
I(0, q) is J(q) to the bit, which makes Ghat(xi, 0) zero."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_lattice_forms(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    exe = tmp_path / "radial_lattice_check"
    subprocess.run([gxx, "-std=c++17", "-O2", "-o", str(exe), os.path.join(HERE, "host", "radial_lattice_check.cpp")],
                   check=True, capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout.split("\n")
    rows = [r.split() for r in out if r.strip()]
    assert len(rows) == 8
    for r in rows:
        assert float(r[2]) <= 12 and float(r[3]) <= 12 and int(r[4]) == 0, r
