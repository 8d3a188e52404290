"""The size rule of the sweep's work tiles, compiled for the CPU: a call is cut
into enough tiles that no thread block is left with a single one, at every
dimension's block width."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1409_3901_gb300", "csrc")
PROGRAM = r"""
#include <stdint.h>
#include <stdio.h>
#define __host__
#define __device__
#include "td_internal.h"
int main(void)
{
    int d, n, sms;
    long long total;
    while (scanf("%d %d %lld %d", &d, &n, &total, &sms) == 4)
        printf("%d %d %d %d %d %d\n", td_auto_spw(d, n, total, sms), td_sweep_warps(d), TD_TILE_WARPS,
               td_tuned_spw(d, n, total, sms, 0), td_tuned_spw(d, n, total, sms, 1024), td_tuned_spw(d, n, total, sms, 16));
    return 0;
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("tile")
    (d / "rule.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(d / "rule.cpp"), "-o", str(d / "rule")])

    def call(rows):
        text = "\n".join("%d %d %d %d" % r for r in rows)
        out = subprocess.run([str(d / "rule")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return call


def test_three_tiles_and_more_for_every_resident_block(rule):
    g = np.random.default_rng(3)
    rows = [(int(d), int(n), int(10 ** t), int(s)) for d, n, t, s in
            zip(g.integers(3, 7, 4000), np.exp(g.uniform(1, 7.6, 4000)), g.uniform(2, 14, 4000),
                g.choice([40, 132, 152], 4000))]
    for (d, n, total, sms), (spw, warps, tile_warps, *_) in zip(rows, rule(rows)):
        resident = sms * (16 // warps)
        assert 2 <= spw <= 2048
        assert spw == 2 or spw * tile_warps * n * 3 * resident <= total
        assert spw == 2 or spw * n <= 2 ** 19


def test_a_tuned_size_holds_in_calls_of_many_tiles(rule):
    """24 tiles of the tuned size and more a block, or the size rule's."""
    g = np.random.default_rng(4)
    rows = [(int(d), int(n), int(10 ** t), 152) for d, n, t in
            zip(g.integers(3, 7, 4000), np.exp(g.uniform(1, 7.6, 4000)), g.uniform(2, 16, 4000))]
    seen = set()
    for (d, n, total, sms), (spw, warps, tile_warps, none, large, small) in zip(rows, rule(rows)):
        work = tile_warps * n * 24 * sms * (16 // warps)  # of 24 tiles a block, per subset and warp
        assert none == spw
        for tuned, got in ((1024, large), (16, small)):
            if tuned <= spw or tuned * work <= total:
                assert got == tuned
            else:
                assert got == max(spw, total // work)
            seen.add((tuned <= spw, tuned * work <= total))
    assert len(seen) == 4


def test_a_call_without_points_or_work_has_a_size(rule):
    assert [r[0] for r in rule([(3, 0, 0, 152), (6, 1, 0, 152), (0, 5, 10, 152), (2, 2048, 0, 1)])] == [2, 2, 2, 2]


def test_a_scratch_of_so_many_warps_is_used_at_every_block_width(tmp_path):
    """The allocation-free call's scratch holds 640 warps: a kernel of narrow
    blocks gets more blocks, not fewer warps, and never more than are there."""
    src = PROGRAM.replace('"td_internal.h"', '"td_internal.h"\n#define main unused').replace(
        "    return 0;\n}\n", "    return 0;\n}\n#undef main\n"
        "int main(void)\n{\n    for (int d = 2; d <= 6; ++d)\n"
        "        for (int sms = 1; sms <= 152; sms += 151)\n            for (int occ = 1; occ <= 8; ++occ)\n"
        '                printf("%d %d %d %d\\n", sms, occ, td_capped_grid(d, sms, occ, 640), td_sweep_warps(d));\n'
        "    return 0;\n}\n")
    (tmp_path / "grid.cpp").write_text(src)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(tmp_path / "grid.cpp"), "-o", str(tmp_path / "grid")])
    rows = [tuple(map(int, line.split())) for line in
            subprocess.check_output([str(tmp_path / "grid")], text=True).splitlines()]
    assert len(rows) == 80
    for sms, occ, grid, warps in rows:
        assert grid <= sms * occ and grid * warps <= 640
        assert grid == sms * occ or grid * warps == 640
