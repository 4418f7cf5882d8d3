"""Host check of the double-precision sums and transport differences formed on the integer
pipes (paper_2502_16818_gb300/csrc/cdbm_exact.h) against the double operations they stand
for: no bit may differ."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2502_16818_gb300", "csrc")


def test_integer_forms_have_the_bits_of_double_arithmetic(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "exact_check")
    subprocess.run([cxx, "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", CSRC, os.path.join(HERE, "exact_check.cc"), "-o", exe],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    v = dict(zip(r.stdout.split()[::2], map(int, r.stdout.split()[1::2])))
    assert v == {"nnd": 0, "sums": 0, "float": 0, "taken": 0}, r.stdout
