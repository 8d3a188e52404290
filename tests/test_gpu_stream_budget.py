"""Admission to the request stream counts every array that grows with the
queries."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# per query: its point (6 words), its dataset, its place in the work order, the
# 104-byte record, five 8-byte tile prefixes, tile size, minimum and result
PER_QUERY = 24 + 4 + 4 + 104 + 40 + 4 + 4 + 4


def test_a_budget_below_the_queries_arrays_is_refused():
    from paper_1409_3901_gb300 import tukey
    g = np.random.default_rng(6)
    x = g.integers(-9, 10, (8, 2)).astype(np.int32)
    z = g.integers(-9, 10, (20000, 2)).astype(np.int32)
    ctx = tukey.Context(0)
    need = len(z) * PER_QUERY + x.nbytes
    assert ctx.stream(mem_budget_bytes=need - 1).submit(x, z) is None
    s = ctx.stream(mem_budget_bytes=need + 4096)
    t = s.submit(x, z)
    assert t is not None
    assert np.array_equal(s.wait(t, timeout_us=60_000_000), tukey.Context(0).depth(x, z))
