"""td_stats.filtered_points and exact_points: the points of the passes made for
one subset, certified or not.  The subsets that shared tables decide have no
such pass and add to neither."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _call(p, n, m, **options):
    from paper_1409_3901_gb300 import tukey
    g = np.random.default_rng([p, n, m])
    x = np.rint(40 * g.standard_normal((n, p))).astype(np.int32)
    z = g.integers(-30, 31, (m, p)).astype(np.int32)
    z = z[~(z[:, None] == x[None]).all(axis=2).any(axis=1)]  # every point of every query is nonzero
    ctx = tukey.Context(0, **options)
    ctx.depth(x, z)
    return ctx.last_stats


# rows so short that no run of subsets pays for tables
@pytest.mark.parametrize("p,n", [(2, 500), (3, 20), (4, 12), (5, 11), (6, 10)])
def test_a_pass_for_every_subset_counts_every_point(p, n):
    st = _call(p, n, 12)
    assert st.sweeps > 0 and st.filtered_points + st.exact_points == st.sweeps * n
    # the subset's own p - 2 points have no direction to certify
    assert st.exact_points >= (p - 2) * st.sweeps


@pytest.mark.parametrize("p,n", [(3, 1000), (4, 300), (5, 90)])
def test_subsets_decided_by_tables_count_no_points(p, n):
    # tiles long enough for runs that pay for tables (the size rule cuts a call this small into 16s at p = 3)
    st = _call(p, n, 12, subsets_per_warp=256)
    points = st.filtered_points + st.exact_points
    assert points % n == 0 and 0 < points < st.sweeps * n
    assert st.exact_points >= (p - 2) * (points // n)


def test_the_plain_form_certifies_nothing():
    from paper_1409_3901_gb300 import tukey
    st = _call(4, 40, 4, mode=tukey.TD_MODE_PLAIN_EXACT)
    assert st.filtered_points == 0 and st.exact_points == st.sweeps * 40
