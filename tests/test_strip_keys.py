"""The middle of two strip keys, compiled for the CPU with the compiler's
overflow check: the keys are bit patterns near those of 1.5 * 2^16 and
1.5 * 2^17, whose sum does not fit a signed 32-bit integer."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1409_3901_gb300", "csrc")
PROGRAM = r"""
#include <stdint.h>
#include <stdio.h>
#include <string.h>
#define __host__
#define __device__
#include "td_internal.h"
static int bits(float f)
{
    int v;
    memcpy(&v, &f, 4);
    return v;
}
int main(void)
{
    const float base[2] = { 98304.0f, 196608.0f };
    for (int k = 0; k < 2; ++k)
        for (int a = -128; a < 128; ++a)
            for (int b = a; b < 128; ++b) {
                const int m = bits(base[k]), x = td_key_middle(m + a, m + b);
                if (x - m != (a + b - (((a + b) % 2) + 2) % 2) / 2) return 1;
            }
    printf("ok\n");
    return 0;
}
"""


def test_the_middle_of_two_keys_has_no_overflow(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "keys.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-fsanitize=signed-integer-overflow", "-fno-sanitize-recover=all",
                           "-I", CSRC, str(tmp_path / "keys.cpp"), "-o", str(tmp_path / "keys")])
    assert subprocess.check_output([str(tmp_path / "keys")], text=True) == "ok\n"


def test_the_strips_take_their_middle_from_it():
    with open(os.path.join(CSRC, "td_fan.cuh")) as f:
        code = f.read()
    assert "x1 = td_key_middle(x0, x2)" in code and "(x0 + x2)" not in code
