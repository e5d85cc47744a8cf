"""Division of a float vector by its length near 1
(paper_2203_09467_gb300/csrc/emt_unit.cuh, the mixed-precision field
transport's renormalisation) compiled as host code and compared bit for bit
with sqrtf and the C division: every squared length of its range, the
estimate moved by up to two units of its last place, random components and
components next to the length."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_unit_division_equals_ieee(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "unit_host")
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-o", exe,
                           os.path.join(HERE, "csrc", "unit_host.cpp")])
    out = subprocess.run([exe, "400"], capture_output=True, text=True).stdout
    checked, wrong = (int(v) for v in out.split()[-2:])
    assert checked > 5e7 and wrong == 0, out
