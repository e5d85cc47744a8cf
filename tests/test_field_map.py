"""The FP64 field map (paper_2203_09467_gb300/csrc/emt_field.cuh) compiled as
host code: its error over 1 to 100 substeps of turns from 0.002 to 0.5, along
each axis and in any direction, against the RK4 stages in 113-bit arithmetic,
beside the error of the stages in FP64."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
UNIT = 2.0 ** -53  # half a unit of the last place of 1


def test_field_map_is_as_accurate_as_the_stages(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "field_host")
    subprocess.check_call([cxx, "-O2", "-std=gnu++17", "-ffp-contract=off", "-o", exe,
                           os.path.join(HERE, "csrc", "field_host.cpp")])
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    rows = np.array([[float(v) for v in line.split()] for line in out.splitlines()])
    assert len(rows) == 11 * 5 * 4
    t, n = rows[:, 0], rows[:, 1]
    # Rounding the map's coefficients once, by up to half a unit, turns n
    # substeps by up to n t UNIT too far (the stages round each turn anew): the
    # direction by as much, the position by its integral over the path n t
    # plus half a unit of the path itself.
    turn = n * t * UNIT
    shift = n * t * (1 + n * t / 2) * UNIT
    for name, at, extra in (("position", 3, shift), ("direction", 5, turn)):
        rms, most, stage_rms, stage_most = rows[:, at], rows[:, at + 1], rows[:, at + 4], rows[:, at + 5]
        # the largest of 150 errors scatters by about a quarter of itself from
        # sample to sample
        bad = (rms > 1.1 * stage_rms + extra) | (most > 1.5 * stage_most + 2 * extra)
        assert not bad.any(), f"{name}:\n" + "\n".join(out.splitlines()[i] for i in np.nonzero(bad)[0])
