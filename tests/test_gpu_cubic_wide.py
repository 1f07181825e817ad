"""Wide intervals: one call over them gives what calls over narrow parts give
(the forms of a window are found near both of its ends, whatever its width)."""
import numpy as np
import pytest

import paper_2507_06579_gb300 as E

pytestmark = pytest.mark.gpu

BLOCK = 1 << 24


@pytest.fixture(scope="module")
def ctx():
    E.build()
    c = E.Context(0)
    yield c
    c.close()


def test_one_wide_count_is_the_sum_of_its_blocks(ctx):
    hi = 10**10
    lo = [5] + list(range(BLOCK, hi, BLOCK))
    p = ctx.plan_create(lo, lo[1:] + [hi])
    p.launch()
    want = int(p.counts().sum())
    p.destroy()
    assert ctx.count_range(5, hi) == want == ctx.pi_E(hi - 1)


@pytest.mark.parametrize("lo,width", [(5, 13 * 10**8), (930_189, 10**9), (2 * 10**9 + 3, 8 * 10**9)])
def test_wide_bitmaps_are_those_of_their_parts(ctx, lo, width):
    hi = lo + width
    f, s, _ = ctx.classify_range(lo, hi)
    part = 256 << 18  # 2^23 candidates, whole words
    for a in range(lo, hi, part):
        w = (a - lo) // 256
        fp, sp, _ = ctx.classify_range(a, min(hi, a + part))
        assert np.array_equal(f[w:w + len(fp)], fp) and np.array_equal(s[w:w + len(sp)], sp)
