"""The server's lane search (taken at the default giant_after): counts equal
those of the range call over ranges of one and of several rounds, on both
quotients and below the search's least d, and a server whose budget has no
room for the search's tables gives the same answers by walking."""
import pytest

import paper_2507_06579_gb300 as E

pytestmark = pytest.mark.gpu

RANGES = [(5, 2_000_005), (10**9, 10**9 + 400_000),
          (10**10 + 3, 10**10 + 3 + 8 * ((1 << 19) + 77)),    # more than one round of survivors
          (10**12 - 10**6, 10**12 + 7), (4390000000000 - 10**5, 4390000000000 + 10**5),
          (E.EIS_D_LIMIT - 50_000, E.EIS_D_LIMIT), (10**11, 10**11 + 8), (10**11, 10**11)]


@pytest.mark.parametrize("budget", [0, 256 << 20], ids=["search", "no_room"])
def test_counts_equal_the_range_call(budget):
    E.build()
    with E.Context(0) as ctx:
        want = [ctx.count_range(lo, hi) for lo, hi in RANGES]
    with E.Context(0, mem_budget_bytes=budget) as c:
        used0 = c.get_option(E.EIS_OPT_MEM_IN_USE)
        with E.Server(c, slots=2) as srv:
            assert (srv.stats()["reserved_bytes"] > (1 << 30)) == (budget == 0)
            for _ in range(2):  # the slots' tables are used again
                ids = [srv.submit_count(lo, hi) for lo, hi in RANGES]
                assert [srv.wait(i)[:2] for i in ids] == [(E.EIS_OK, n) for n in want]
        assert c.get_option(E.EIS_OPT_MEM_IN_USE) == used0
