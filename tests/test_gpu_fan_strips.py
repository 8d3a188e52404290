"""The shared tables of long fans (subsets with a common tail) on the GPU:
tiles that hold whole fans, several for every team, and more than one tile a
query, so that the bounds are tested against a finite minimum, in more than
one round of strips and with more strips than the first fans take.

Against the plain exact form, which shares none of it.  Counts are integers:
equality, no tolerance.  td_stats says that the tables decided something: a
subset they decide has no pass over the points."""
from math import comb

import numpy as np
import pytest

from test_gpu_fan import _data

pytestmark = pytest.mark.gpu


def _check(p, n, kind, spw, **options):
    from paper_1409_3901_gb300 import tukey
    x, z = _data(tukey, kind, n, p, 3)
    want = tukey.Context(0, mode=tukey.TD_MODE_PLAIN_EXACT, **options).depth(x, z)
    ctx = tukey.Context(0, subsets_per_warp=spw, **options)
    assert np.array_equal(ctx.depth(x, z), want)
    if kind == "uniform":
        st = ctx.last_stats
        nonzero = min(int((x != q).any(axis=1).sum()) for q in z)
        assert st.filtered_points + st.exact_points < st.sweeps * nonzero


# teams of 1 (packed and unpacked tables), 2, 4 and 8 warps; a tile is 8 spw subsets
@pytest.mark.parametrize("kind", ["uniform", "ties", "wide"])
@pytest.mark.parametrize("p,n,spw", [(3, 255, 256), (3, 257, 256), (3, 1000, 128), (3, 2048, 64), (3, 2048, 256),
                                     (4, 255, 1024), (4, 257, 1024), (4, 383, 256), (4, 385, 2048), (4, 770, 256),
                                     (4, 1538, 1024), (5, 113, 2048), (5, 257, 1024)])
def test_whole_queries_in_long_tiles(p, n, spw, kind):
    _check(p, n, kind, spw)


# many points on one span make the exact form of every subset in it cubic in
# their number and worse: short rows
@pytest.mark.parametrize("p,n,spw", [(3, 257, 256), (4, 255, 1024), (4, 257, 1024)])
def test_points_on_few_lines(p, n, spw):
    _check(p, n, "lines", spw)


@pytest.mark.parametrize("kind", ["uniform", "ties", "wide"])
@pytest.mark.parametrize("p,n,spw", [(4, 2047, 1024), (5, 578, 512), (5, 1153, 1024), (6, 120, 1024), (6, 257, 512),
                                     (6, 770, 256), (6, 1538, 256)])
def test_ranges_of_several_long_tiles(p, n, spw, kind):
    """Without the seed, so that the minimum is the range's own."""
    shards = comb(n, p - 2) // (24 * spw)  # three tiles a query
    for index in (0, shards // 2, shards - 1):
        _check(p, n, kind, spw, unseeded=True, shard_index=index, shard_count=shards)
