"""A plan captured into a caller's CUDA graph: each replay is a full pass whose
results the plan reads."""
import numpy as np
import pytest

import paper_2507_06579_gb300 as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,n", [(10**6, 5_000), (10**10, 1 << 20)])
def test_replays_give_the_plans_results(lo, n):
    torch = pytest.importorskip("torch")
    E.build()
    with E.Context(0) as c:
        want = c.count_range(lo, lo + 8 * n)
        f, s, _ = c.classify_range(lo, lo + 8 * n)
        c.set_option(E.EIS_OPT_USE_GRAPH, 0)
        p = c.plan_create([lo], [lo + 8 * n])
        p.launch()
        p.counts()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            p.launch(torch.cuda.current_stream())
        for _ in range(2):
            g.replay()
            torch.cuda.synchronize()
            assert int(p.counts()[0]) == want
            pf, ps = p.copy_bitmaps()
            assert np.array_equal(pf, f) and np.array_equal(ps, s)
        torch.cuda.synchronize()
        p.destroy()
