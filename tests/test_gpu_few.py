"""The library's own search settings for plans of few d (longer recording
walks, denser tables): codes and classes equal the walk's to the centre, over
the factors the rule can give and up to the largest d."""
import pytest

import paper_2507_06579_gb300 as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,n", [
    (6 * 10**8, 140_001),            # the smallest d that are searched
    (10**10 + 1, 12_000),            # factor 2.8, then 1.4, then none
    (10**10 + 1, 300_001), (10**10 + 1, 700_001),
    (10**12, 1_501), (4_390_000_000_000 - 4_000, 9_001),  # across the quotients' border
    (E.EIS_D_LIMIT - 8 * 20_000, 20_000)])
def test_few_d_equal_the_walk(lo, n):
    E.build()
    hi = min(lo + 8 * n, E.EIS_D_LIMIT)
    got = []
    for limit in (1 << 26, 1 << 25):  # own settings; every d walked
        with E.Context(0) as ctx:
            ctx.set_option(E.EIS_OPT_STEP_LIMIT, limit)
            p = ctx.plan_create([lo], [hi], E.EIS_MODE_PERSISTENT, E.EIS_PLAN_CLASSES)
            p.launch()
            flags, sq = p.copy_bitmaps()
            deferred = p.stats()["deferred"]
            p.destroy()
            got.append((flags.tobytes(), sq.tobytes(), ctx.class_counts(lo, hi),
                        ctx.classify_range_log(lo, hi).tobytes()))
        assert (deferred > 0) == (limit == 1 << 26)
    assert got[0] == got[1]
