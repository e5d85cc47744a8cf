"""Stack that the allocation-free entry point takes from its caller's thread,
as the host compiler reports it: the largest geometry's planes (32 KB) and a
few kilobytes more, so that threads with small stacks can call it."""
import os
import re
import subprocess

from paper_2203_09467_gb300 import build


def test_static_entry_point_fits_a_small_stack(tmp_path):
    flags = [f + ",-fstack-usage" if f.startswith("-fPIC") else f for f in build.COMMON]
    subprocess.check_call([build.nvcc(), *build.ARCH, *flags, "-c", os.path.join(build.CSRC, "emt_api.cu"),
                           "-o", str(tmp_path / "emt_api.o")], cwd=tmp_path, stderr=subprocess.DEVNULL)
    lines = "".join((tmp_path / f).read_text() for f in os.listdir(tmp_path) if f.endswith(".su")).splitlines()
    frame = [int(re.search(r"\t(\d+)\t", line).group(1)) for line in lines if "emt_transport_static(" in line]
    assert len(frame) == 1 and frame[0] <= 64 * 1024, frame
