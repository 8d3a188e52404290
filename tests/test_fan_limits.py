"""The limits that the sweep's fans rely on are asserted where the kernels are
compiled: a wider spread or longer rows stop the build instead of dropping
subsets."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1409_3901_gb300", "csrc")


def _asserts():
    with open(os.path.join(CSRC, "td_fan.cuh")) as f:
        code = f.read()
    found = []
    at = code.find("static_assert(")
    while at >= 0:
        text = code[at:code.index(");", at) + 2]
        if "a warp's blocks" in text:
            found.append(text)
        at = code.find("static_assert(", at + 1)
    return found


@pytest.mark.parametrize("spread,rows,holds", [(96, 2048, True), (128, 2048, True), (129, 2048, False),
                                               (96, 4096, True), (96, 4097, False)])
def test_flags_of_a_warps_blocks(tmp_path, spread, rows, holds):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    asserts = _asserts()
    assert len(asserts) == 2
    (tmp_path / "a.cpp").write_text('#define __host__\n#define __device__\n#include "td_internal.h"\n'
                                    "#define TD_FAN_SPREAD %d\n#define TD_MAX_N %d\n" % (spread, rows) +
                                    "\n".join(asserts) + "\n")
    rc = subprocess.run(["g++", "-std=c++17", "-fsyntax-only", "-I", CSRC, str(tmp_path / "a.cpp")],
                        capture_output=True).returncode
    assert (rc == 0) == holds
