"""Plans whose d are decided by cubic forms (k_cubic) give what the walk
gives: against the oracle where it can walk, else against the same context
with a lowered step limit, which walks every d."""
import numpy as np
import pytest

import paper_2507_06579_gb300 as E
from paper_2507_06579_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    E.build()
    c = E.Context(0)
    yield c
    c.close()


class _walking:
    """The block's plans walk every d (step limit below its default)."""

    def __init__(self, ctx):
        self.ctx = ctx

    def __enter__(self):
        self.ctx.set_option(E.EIS_OPT_STEP_LIMIT, 1 << 25)

    def __exit__(self, *exc):
        self.ctx.set_option(E.EIS_OPT_STEP_LIMIT, 1 << 26)


@pytest.mark.parametrize("lo,n", [(10**9 - 777, (1 << 18) + 37), (3 * 10**8 + 11, 400_001)])
def test_codes_and_classes_match_oracle(ctx, orc, lo, n):
    """Several tiles and a ragged tail, every candidate."""
    hi = lo + 8 * n
    ref = orc.classify_range(lo, hi, thetas=True)
    codes, cnt = ctx.classify_range_u8(lo, hi)
    steps = ctx.stats()["baby_steps"]
    assert np.array_equal(codes, ref["codes"]) and cnt == int((ref["codes"] == 2).sum())
    assert np.array_equal(ctx.classify_range_log(lo, hi), ref["thetas"])
    with _walking(ctx):
        ctx.count_range(lo, hi)
        assert 5 * steps < ctx.stats()["baby_steps"]  # the forms decided most d


@pytest.mark.parametrize("lo,hi", [
    W.CFG_TOP, (5, 10**9 + 1),
    (10**12 - 10**7 - 3, 10**12 + 5),
    (4390000000000 - 3 * 10**6, 4390000000000 + 10**6),   # across the fast quotient's limit
    (E.EIS_D_LIMIT - 2 * 10**6 - 5, E.EIS_D_LIMIT),
])
def test_bitmaps_equal_the_walk(ctx, lo, hi):
    f, s, c = ctx.classify_range(lo, hi)
    steps = ctx.stats()["baby_steps"]
    with _walking(ctx):
        f0, s0, c0 = ctx.classify_range(lo, hi)
        assert 5 * steps < ctx.stats()["baby_steps"]
    assert c == c0 and np.array_equal(f, f0) and np.array_equal(s, s0)


@pytest.mark.parametrize("flags", [0, E.EIS_PLAN_CLASSES, E.EIS_PLAN_PRIMES,
                                   E.EIS_PLAN_CLASSES | E.EIS_PLAN_PRIMES])
@pytest.mark.parametrize("nbaby", [0, 512])
def test_mixed_plan_equals_the_walk(ctx, flags, nbaby):
    """Intervals the forms decide beside others that are walked (short, empty,
    overlapping), with the lane search and without, launched twice."""
    lo, hi = W.batched_intervals(n=60, seed=21, a_range=(1e6, 1e11), len_range=(1e2, 1e5))
    lo = [int(x) for x in lo] + [0, 5, 10**10, 10**10 + 10**6, 2 * 10**11, 3 * 10**9]
    hi = [int(x) for x in hi] + [0, 6, 10**10 + 4 * 10**6, 10**10 + 3 * 10**6 + 9, 2 * 10**11 + 2 * 10**6,
                                 3 * 10**9 + 2 * 10**7 + 1]
    ctx.set_option(E.EIS_OPT_GIANT_THRESHOLD, nbaby)
    try:
        got = []
        for walk in (False, True):
            if walk:
                ctx.set_option(E.EIS_OPT_STEP_LIMIT, 1 << 25)
            p = ctx.plan_create(lo, hi, E.EIS_MODE_PERSISTENT, flags)
            out = []
            for _ in range(2):
                p.launch()
                out += [p.counts(), p.counts_D(), *p.copy_bitmaps()]
                if flags & E.EIS_PLAN_CLASSES:
                    out.append(p.class_counts())
            got.append((out, p.stats()["baby_steps"]))
            p.destroy()
    finally:
        ctx.set_option(E.EIS_OPT_GIANT_THRESHOLD, 0)
        ctx.set_option(E.EIS_OPT_STEP_LIMIT, 1 << 26)
    assert all(np.array_equal(a, b) for a, b in zip(got[0][0], got[1][0]))
    assert got[0][1] < got[1][1]


def test_no_room_for_the_second_bitmap_walks(orc):
    """A budget that holds the plan but not the forms' bitmap: the plan is
    made all the same, and counts alike."""
    lo, n = 10**9, 1 << 20
    walk = [(E.EIS_D_LIMIT, 0, 16)]  # no search, whose pool would take what room there is
    with E.Context(0) as c:
        c.set_tune_table(walk)
        used0 = c.get_option(E.EIS_OPT_MEM_IN_USE)
        p = c.plan_create([lo], [lo + 8 * n])
        need = c.get_option(E.EIS_OPT_MEM_IN_USE) - used0
        p.launch()
        want = int(p.counts()[0])
        p.destroy()
    with E.Context(0, mem_budget_bytes=used0 + need - 64) as c:
        c.set_tune_table(walk)
        p = c.plan_create([lo], [lo + 8 * n])
        p.launch()
        assert int(p.counts()[0]) == want
        p.destroy()
        assert c.get_option(E.EIS_OPT_MEM_IN_USE) == used0
