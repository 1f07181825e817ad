"""The square-free sieve with its primes split between the tiles' kernel and
the intervals' (k_sieve_big): bitmaps against the oracle's range sieve where
the split begins (512^2), where it is first used, with several intervals in a
plan, ragged ends, and up to the table's last prime."""
import numpy as np
import pytest

import paper_2507_06579_gb300 as E

pytestmark = pytest.mark.gpu


def _sqfree(lo, hi):
    """Square-freeness of every candidate by trial division with odd k."""
    d = np.arange(lo + (13 - lo % 8) % 8, hi, 8, dtype=np.int64)
    ok = np.ones(len(d), np.uint8)
    top = int(np.sqrt(float(hi))) + 1
    for k in range(3, top + 1, 2):
        k2 = k * k
        first = (-int(d[0])) * pow(8, -1, k2) % k2  # d0 + 8 i == 0 (mod k^2)
        ok[first::k2] = 0
    return ok


@pytest.mark.parametrize("lo,n", [
    (5, 70_001), (512 * 512 * 5 - 400, 3_000), (10**7, 65_536), (18_000_000, 65_537),
    (10**9 + 11, 131_075), (10**12 - 8 * 20_000, 20_000), (E.EIS_D_LIMIT - 8 * 3_000 - 3, 3_000)])
def test_square_free_bitmap(lo, n):
    E.build()
    hi = min(lo + 8 * n, E.EIS_D_LIMIT)
    ref = _sqfree(lo, hi)
    with E.Context(0) as ctx:
        for mode in (E.EIS_MODE_PERSISTENT, E.EIS_MODE_PLAIN):
            # beside two other intervals, one of them empty
            p = ctx.plan_create([lo, 0, 3 * 10**8], [hi, 0, 3 * 10**8 + 999], mode)
            p.launch()
            _, sq = p.copy_bitmaps()
            off = int(p.bitmaps()[2][0])
            assert int(p.counts_D()[0]) == int(ref.sum())
            bits = np.unpackbits(sq[off:].view(np.uint8), bitorder="little")[:len(ref)]
            p.destroy()
            assert np.array_equal(bits, ref)


@pytest.mark.parametrize("lo,n", [(5, 8_191), (10**9, 8_193), (10**10, 98_304), (10**9, 1_245_185)])
def test_short_tiles(lo, n):
    """A small plan's shorter tiles give what whole ones give (a context
    without room for the longer tile table), classes and counts included."""
    E.build()
    got = []
    with E.Context(0) as ctx:
        used0 = ctx.get_option(E.EIS_OPT_MEM_IN_USE)
    for budget in (0, used0 + (1 << 20) + 12 * n):
        with E.Context(0, budget) as ctx:
            p = ctx.plan_create([lo, lo + 8 * n + 64], [lo + 8 * n, lo + 8 * n + 800],
                                E.EIS_MODE_PERSISTENT, E.EIS_PLAN_CLASSES)
            p.launch()
            flags, sq = p.copy_bitmaps()
            got.append((flags.tobytes(), sq.tobytes(), p.counts().tolist(), p.counts_D().tolist(),
                        p.class_counts().tolist()))
            p.destroy()
    assert got[0] == got[1]
