"""The query's running minimum that the warps of a sweep share.

Warps lower it while others read it, and what is decided from it (which
subsets are swept again) guards full-warp operations: every lane of a warp has
to decide alike, so a warp takes the value one lane read."""
import glob
import os
import re

import numpy as np
import pytest

import oracle

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1409_3901_gb300", "csrc")


def _code():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"/\*.*?\*/|//[^\n]*", "", f.read(), flags=re.S)


def test_no_lane_decides_from_a_read_of_its_own():
    """A read of the minimum while other warps lower it goes to one thread
    (s_qmin, read by thread 0 and shared after a barrier) or through TdQmin,
    whose value leaves it by a shuffle from lane 0."""
    reads = []
    for name, code in _code():
        struct = re.search(r"struct TdQmin \{.*?\n\};", code, re.S)
        if struct:
            assert re.search(r"int get\(\) const \{ return __shfl_sync\(TD_FULL, v, 0\); \}", struct.group(0))
            code = code.replace(struct.group(0), "")
            names = re.findall(r"TdQmin (\w+)", code)
            assert names and not any(re.search(r"\b%s\.v\b" % n, code) for n in names)
        reads += [(name, line.strip()) for line in code.splitlines()
                  if re.search(r"volatile[^;]*\bqmin", line) or re.search(r"__ldcg|ld\.(volatile|relaxed)[^;]*qmin", line)]
    assert [line.split("=")[0].strip() for _, line in reads] == ["s_qmin"], reads


@pytest.mark.gpu
@pytest.mark.parametrize("p,n,spw", [(3, 500, 2), (4, 120, 2), (4, 120, 64), (5, 40, 2), (6, 24, 2)])
def test_counts_hold_while_the_minimum_falls(p, n, spw):
    """No upper bound to begin with and small tiles: many warps lower the
    minimum at once, in another order every time."""
    from paper_1409_3901_gb300 import tukey
    g = np.random.default_rng([p, n])
    x = np.rint(40 * g.standard_normal((n, p))).astype(np.int32)
    z = np.concatenate([x[:1], np.rint(np.median(x, axis=0, keepdims=True)).astype(np.int32)])
    want = oracle.depth_many(x, z)
    ctx = tukey.Context(0, unseeded=True, subsets_per_warp=spw)
    for _ in range(30):
        assert np.array_equal(ctx.depth(x, z), want)
