"""The sweep of whole fans (subsets with a common tail) on the GPU, at the
sizes where its forms change: rows around multiples of 32 and 64 points, the
byte-packed tables' limit of 255 points, every team size (rows of 384, 768 and
1536 points at p = 4, 576 at p = 5, 768 at p = 6), fans cut by a shard's ends,
and coordinates that take each arithmetic of the projection.

Small rows against the CPU oracle; longer ones over ranges of subset positions
against the plain exact form, which shares none of it.  Counts are integers:
equality, no tolerance."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def td():
    from paper_1409_3901_gb300 import tukey
    return tukey


def _data(tukey, kind, n, p, seed):
    g = np.random.default_rng([n, p, seed])
    lim = {"uniform": 127, "ties": 3, "wide": int(tukey.td_coord_limit(p)) // 2, "lines": 40}[kind]
    x = g.integers(-lim, lim + 1, (n, p))
    if kind == "lines":  # most rows on three lines through one data row, the last coordinate often zero
        step = g.integers(-1, 2, (3, p))
        k = 2 * n // 3
        x[:k] = g.integers(-lim // 2, lim // 2, (k, 1)) * step[g.integers(0, 3, k)] // 2
        x[::3, p - 1] = 0
    x = x.astype(np.int32)
    mid = (x[g.integers(0, n, 1)] // 2).astype(np.int32)
    return x, np.concatenate([x[g.integers(0, n, 2)], mid]).astype(np.int32)


@pytest.mark.parametrize("kind", ["uniform", "ties", "wide", "lines"])
@pytest.mark.parametrize("p,n", [(3, 4), (3, 32), (3, 33), (3, 65), (4, 6), (4, 31), (4, 64), (4, 65), (5, 9), (5, 33),
                                 (6, 8), (6, 21)])
def test_small_rows_match_the_oracle(td, p, n, kind):
    x, z = _data(td, kind, n, p, 1)
    want = oracle.depth_many(x, z)
    assert np.array_equal(td.Context(0).depth(x, z), want)
    assert np.array_equal(td.Context(0, early_exit=True).depth(x, z), want)


@pytest.mark.parametrize("kind", ["uniform", "ties", "wide", "lines"])
@pytest.mark.parametrize("p,n", [(3, 255), (3, 257), (3, 2048), (4, 255), (4, 256), (4, 383), (4, 384), (4, 767),
                                 (4, 769), (4, 1536), (4, 2047), (5, 113), (5, 255), (5, 256), (5, 577), (6, 120),
                                 (6, 257), (6, 769)])
def test_ranges_match_the_plain_form(td, p, n, kind):
    x, z = _data(td, kind, n, p, 2)
    total = 1
    for i in range(p - 2):
        total = total * (n - i) // (i + 1)
    shards = max(1, total // (3000 if p < 6 else 800))
    for index in sorted({0, shards // 3, shards - 1}):
        opts = {"shard_index": index, "shard_count": shards, "unseeded": True}
        want = td.Context(0, mode=td.TD_MODE_PLAIN_EXACT, **opts).depth(x, z)
        assert np.array_equal(td.Context(0, **opts).depth(x, z), want)
