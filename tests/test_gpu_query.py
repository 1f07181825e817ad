"""k_query (one membership query in one launch) against the range path and the
oracle: where the period ends in the baby walk, just past it, in the first 32
giant steps, in the block's first round and later, on both quotients."""
import numpy as np
import pytest

import paper_2507_06579_gb300 as E

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    E.build()
    c = E.Context(0)
    yield c
    c.close()


def _ask(ctx, d):
    try:
        return 2 if ctx.is_eisenstein(d) else 1
    except E.EisError as e:
        assert e.code == E.EIS_ENOTD, (d, e)
        return 0


@pytest.mark.parametrize("stride", [0, 256, 4096])   # N: automatic, the least, the largest
@pytest.mark.parametrize("lo,n", [(5, 600), (10**5, 300), (10**7, 300), (10**9, 300), (10**11, 200),
                                  (10**12, 150), (2 * 10**12 - 400, 100),          # N 256 | 512
                                  (4390000000000 - 400, 100), (E.EIS_D_LIMIT - 800, 100)])
def test_queries_equal_the_range(ctx, lo, n, stride):
    """Every candidate of a window, square factors included."""
    d0 = lo + ((13 - lo % 8) % 8)
    n = min(n, (E.EIS_D_LIMIT - d0 + 7) // 8)
    codes, _ = ctx.classify_range_u8(d0, min(d0 + 8 * n, E.EIS_D_LIMIT))
    assert len(codes) == n
    ctx.set_option(E.EIS_OPT_GIANT_STRIDE, stride)
    try:
        got = np.array([_ask(ctx, d0 + 8 * k) for k in range(n)], np.uint8)
    finally:
        ctx.set_option(E.EIS_OPT_GIANT_STRIDE, 0)
    assert np.array_equal(got, codes)


def test_periods_around_the_baby_walk_match_oracle(ctx, orc):
    """d whose period is within a few steps of 2N (the centre at the walk's
    end) and of the first giant step, N = 256."""
    near = []
    for d in range(1_000_005, 1_600_000, 8):
        if orc.in_D(d):
            rc, theta, period = orc.walk_mod2(d)
            assert rc == 0
            if any(abs(period - p) <= 12 for p in (512, 640, 768, 1024)):
                near.append((d, theta))
    assert len(near) > 100
    ctx.set_option(E.EIS_OPT_GIANT_STRIDE, 256)
    try:
        for d, theta in near:
            assert ctx.is_eisenstein(d) == (theta == 1), d
    finally:
        ctx.set_option(E.EIS_OPT_GIANT_STRIDE, 0)
