"""Host check of the 64-bit fixed-point arithmetic of the FP64 stage kernels
(paper_2502_16818_gb300/csrc/cdbm_fixed.h) against 113-bit arithmetic.

Bounds: conversions are exact or correctly rounded (0 mismatches).  The general update
rounds its sum once, to half a unit in the last place of the result, which is at most
(2.5 + 1 + 1) times the largest operand -- up to 4 units of 2^-53 of it -- plus one unit
of 2^-58 per converted operand and product.  The form for operands of one exponent rounds
relaxation and transport once each: half a unit, plus the 64ths of the first sum."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2502_16818_gb300", "csrc")


def test_fixed_point_arithmetic(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "fixed_check")
    subprocess.run([cxx, "-O2", "-std=gnu++17", "-I", CSRC, os.path.join(HERE, "fixed_check.cc"), "-o", exe],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    v = dict(zip(r.stdout.split()[::2], map(float, r.stdout.split()[1::2])))
    for name in ("to_double", "round_trip", "used", "ties"):
        assert v[name] == 0, r.stdout
    assert v["any"] <= 4.5, r.stdout
    assert v["fast"] <= 1.0 + 2.0 / 64, r.stdout
