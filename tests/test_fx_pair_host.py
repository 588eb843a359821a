"""The fixed-point pair arithmetic of the FP64 operators on the host, against
long double (tests/fx_pair_check.cpp).

Tolerance, relative to the sum of a row's absolute terms: the kernel tables
are within 2^-50.5 of sigma_i (6.3e-16), the other roundings of a term below
2^-54 each, the conversion of the sum to double 1.1e-16: 1e-15 in all.  The
fused operators share one fixed-point unit between their two layers, so the
smaller layer is held to the larger one's scale."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fixed_point_terms_match_long_double(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path / "fx_pair_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-x", "c++", os.path.join(HERE, "fx_pair_check.cpp"), "-o", exe],
                   check=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    rows = [ln.split() for ln in lines if ln]
    assert len(rows) == 9 * 8
    bad = [r for r in rows if not float(r[1]) <= 1e-15]
    assert not bad, bad
