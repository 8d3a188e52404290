"""The problem that td_autotune times: long enough, by the clock and in tiles,
for the choice to be about the tile size and not about how the last tiles
fall."""
from math import comb

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n", [(4, 300), (4, 1000), (5, 150), (5, 384)])
def test_the_problem_is_long_enough(p, n):
    import torch
    from paper_1409_3901_gb300 import tukey
    r = tukey.Context(0).autotune(p, n)
    # the first problem stays if it is within a quarter of 10 ms, a shorter one is scaled by its own time
    assert 1 <= r["queries"] <= 16384 and r["ms_default"] >= 6.0
    blocks = torch.cuda.get_device_properties(0).multi_processor_count * (2 if p == 4 else 4)
    tile = 8 * min(2048, 2 ** 19 // n)
    assert r["queries"] * comb(n, p - 2) >= 0.8 * 63 * blocks * tile


def test_short_rows_stop_at_the_most_queries():
    from paper_1409_3901_gb300 import tukey
    r = tukey.Context(0).autotune(3, 20)
    assert r["queries"] == 16384 and r["ms_default"] > 0
