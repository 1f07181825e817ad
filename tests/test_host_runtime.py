"""Host side of plans and calls (allocation, ordering between streams, memory
budget), over a CUDA runtime without a device (fakert.py)."""
import pytest

import fakert
import paper_2507_06579_gb300 as E


@pytest.fixture()
def rt():
    with fakert.installed() as L:
        yield L


@pytest.mark.parametrize("flags", [0, E.EIS_PLAN_CLASSES, E.EIS_PLAN_PRIMES])
@pytest.mark.parametrize("thr", [0, 1024])
def test_a_plans_buffers_are_waited_for_before_other_streams_use_them(rt, flags, thr):
    """Buffers are allocated in the order of the context's own stream: the plan
    waits for every one of them before its launches, on any stream, use it."""
    with E.Context(0) as c:
        c.set_option(E.EIS_OPT_GIANT_THRESHOLD, thr)
        for stream in (None, 12345):
            p = c.plan_create([10**9, 10**10], [10**9 + 10**8, 10**10 + 10**8], E.EIS_MODE_PERSISTENT, flags)
            p.launch(stream)
            p.counts()
            p.destroy()
        assert rt.fake_launches(b"k_cubic") > 0  # the forms' bitmap is one of them
        c.count_range(10**9, 10**9 + 10**8)
        c.classify_range_u8(10**9, 10**9 + 10**8)
    assert rt.fake_violations() == 0


def _plan(rt, c, n=1 << 23):
    """Kernels of one launch of a plan of n candidates, or None if it is refused."""
    try:
        p = c.plan_create([10**9], [10**9 + 8 * n])
    except E.EisError as e:
        assert e.code == E.EIS_ENOMEM
        return None
    rt.fake_fail_after(-1, 0)
    p.launch()
    p.counts()
    p.destroy()
    return {k: rt.fake_launches(k.encode()) for k in ("k_cubic", "k_walk_record", "k_walk_persistent")}


def test_a_plan_that_loses_the_forms_is_sized_for_all_its_d(rt):
    """Where the memory for the forms' bitmap cannot be had, the search's rounds
    are those of a plan that never had the forms (they were those of 15% of the
    d, and the last round walked the rest)."""
    def context():
        c = E.Context(0)
        c.set_option(E.EIS_OPT_USE_GRAPH, 0)
        c.set_option(E.EIS_OPT_GIANT_THRESHOLD, 1024)
        c.set_option(E.EIS_OPT_BSGS_CHUNK, 1 << 20)
        return c

    with context() as c:
        c.set_option(E.EIS_OPT_STEP_LIMIT, 1 << 25)  # no forms
        rt.fake_reset()
        without = _plan(rt, c)
    assert without["k_cubic"] == 0 and without["k_walk_record"] == 8
    lost = 0
    for n in range(16):
        with context() as c:
            rt.fake_reset()
            rt.fake_fail_after(n, 2)
            got = _plan(rt, c)
            if got and not got["k_cubic"]:
                assert got == without
                lost += 1
    assert lost > 0


def test_the_warp_search_keeps_its_list_in_a_tight_budget(rt):
    """A budget that holds the plan with the warp search's list but not the
    forms' bitmap: the plan is made, without the forms."""
    def need(limit):
        with E.Context(0) as c:
            c.set_option(E.EIS_OPT_STEP_LIMIT, limit)
            return used(c)

    def used(c):
        c.set_option(E.EIS_OPT_GIANT_KERNEL, E.EIS_GIANT_WARP)
        c.set_option(E.EIS_OPT_GIANT_THRESHOLD, 32768)
        p = c.plan_create([10**9], [10**9 + (8 << 20)])
        n = c.get_option(E.EIS_OPT_MEM_IN_USE)
        p.launch()
        p.destroy()
        return n

    with_forms, without = need(1 << 26), need(1 << 25)
    assert with_forms > without + (1 << 17) - 1  # the bitmap
    with E.Context(0, mem_budget_bytes=with_forms - (1 << 16)) as c:
        rt.fake_reset()
        assert used(c) < with_forms and rt.fake_launches(b"k_cubic") == 0


@pytest.mark.parametrize("thr,n", [(0, 1 << 22), (0, 1 << 17), (1024, 1 << 17)])
def test_without_memory_for_the_searchs_tables_the_plan_walks(rt, thr, n):
    """Callers who did not ask for the search, and small plans, are refused only
    for the buffers a walk needs: two bitmaps, two words a tile, the queue, the
    results and the tables."""
    refused, walked = 0, 0
    for i in range(16):
        with E.Context(0) as c:
            c.set_option(E.EIS_OPT_GIANT_THRESHOLD, thr)
            used0 = c.get_option(E.EIS_OPT_MEM_IN_USE)
            rt.fake_reset()
            rt.fake_fail_after(i, 4)
            try:
                p = c.plan_create([10**12], [10**12 + 8 * n])
            except E.EisError as e:
                assert e.code == E.EIS_ENOMEM
                refused += 1
                p = None
            rt.fake_fail_after(-1, 0)
            if p:
                p.launch()
                p.counts()
                walked += rt.fake_launches(b"k_walk_record") == 0
                p.destroy()
            cached = c.get_option(E.EIS_OPT_MEM_IN_USE) - used0
            assert cached == 0 or rt.fake_launches(b"k_walk_record") > 0  # the kept pool
    assert refused == 7 and walked > 0


def test_the_autotuner_times_the_walk(rt):
    """Three of its trials (the CTA counts) walk every d that the forms leave:
    no trial differs by a setting that its kernels do not use."""
    with E.Context(0) as c:
        rt.fake_reset()
        trials = c.autotune(10**11, 10**11 + (8 << 20))["trials"]
        plans, searched, warp = (rt.fake_launches(k) for k in (b"k_scan_tiles", b"k_walk_record", b"k_giant"))
        assert plans == trials and searched >= 6 and warp == 2
        assert plans - searched - warp == 3
        # and the walk alone can be asked for
        c.set_option(E.EIS_OPT_GIANT_KERNEL, E.EIS_GIANT_WARP)
        assert c.get_option(E.EIS_OPT_GIANT_THRESHOLD) == 0
        rt.fake_reset()
        c.count_range(10**11, 10**11 + (8 << 20))
        assert rt.fake_launches(b"k_walk_persistent") == 1 and rt.fake_launches(b"k_walk_record") == 0


def test_mapped_memory_stays_within_the_budget(rt):
    """Freed buffers that the context keeps mapped count: a plan's search tables
    and a server's slots are not mapped beside them past the budget."""
    budget = 192 << 20
    with E.Context(0, mem_budget_bytes=budget) as c:
        rt.fake_reset()
        walk, search = [(E.EIS_D_LIMIT, 0, 16)], [(E.EIS_D_LIMIT, 512, 16)]
        for rows, n in ((walk, 30 << 20), (search, 1 << 16), (walk, 30 << 20), (walk, 1 << 10)):
            c.set_tune_table(rows)
            p = c.plan_create([10**9], [10**9 + 8 * n])
            p.launch()
            p.counts()
            searched = rt.fake_launches(b"k_walk_record") > 0
            p.destroy()
        assert searched
        with E.Server(c, slots=4, slot_candidates=1 << 22):
            pass
        assert (128 << 20) < rt.fake_peak() <= budget


def test_kept_memory_gives_way_where_the_device_has_no_more(rt):
    """An allocation that the device refuses is tried again without what the
    context keeps mapped: plan buffers, search tables, a server's slots."""
    def grown(c):
        c.set_tune_table([(E.EIS_D_LIMIT, 0, 16)])
        p = c.plan_create([10**9], [10**9 + 8 * (200 << 20)])
        p.launch()
        p.counts()
        p.destroy()
        rt.fake_set_capacity(rt.fake_mapped() + (1 << 20))  # someone else has the rest

    with E.Context(0) as c:
        grown(c)
        c.set_tune_table([(E.EIS_D_LIMIT, 512, 16)])
        p = c.plan_create([10**12], [10**12 + (8 << 18)])  # refused before
        p.destroy()
    rt.fake_set_capacity(200 << 30)
    with E.Context(0) as c:
        grown(c)
        with E.Server(c, slots=1, slot_candidates=1 << 16, giant_after=131072) as srv:  # refused before
            srv.stats()


@pytest.mark.parametrize("rows,lo,search", [
    ([], 10**12, True), ([], 10**6, False),
    ([(10**9, 0, 16)], 10**12, False),   # tuned below 10^9 only: the last row covers every larger d
    ([(10**9, 0, 16), (10**10, 512, 16)], 10**12, True),
    ([(10**9, 512, 16), (10**10, 0, 16)], 10**12, False),
    ([(E.EIS_D_LIMIT, 512, 16)], 10**6, True),
])
def test_a_servers_batch_searches_or_hands_long_walks_on(rt, rows, lo, search):
    """As the tuning row of the batch's largest d says; a batch that walks hands
    its long walks to the giant-step kernel."""
    with E.Context(0) as c:
        c.set_tune_table(rows)
        with E.Server(c, slots=1) as srv:
            rt.fake_reset()
            srv.wait(srv.submit_count(lo, lo + 8000))
            assert (rt.fake_launches(b"k_walk_record") > 0) == search
            assert (rt.fake_launches(b"k_giant") > 0) == (not search)


def test_results_of_a_replayed_plan_are_fetched_again(rt):
    """A launch's results come to the host once; those of a plan that a caller's
    graph replays are waited for and read at every call."""
    with E.Context(0) as c:
        c.set_option(E.EIS_OPT_USE_GRAPH, 0)
        p = c.plan_create([10**9], [10**9 + 8000])

        def waits():
            n = rt.fake_waits()
            p.counts()
            p.copy_bitmaps()
            return rt.fake_waits() - n

        p.launch(777)
        assert waits() == 1 and waits() == 0
        rt.fake_capture(777, 1)
        p.launch(777)
        rt.fake_capture(777, 0)
        assert waits() == 2 and waits() == 2
        p.destroy()
