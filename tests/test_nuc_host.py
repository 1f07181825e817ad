"""The giant steps' product (eis_nuc.cuh) on the host: products of two states
of the principal cycle land on the cycle, with that state's class and third
coefficient, within log d of the sum of the distances; pairs whose norms share
a factor are sent back (kNucRetry), and nothing else fails."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_infra_host import _first_states, _pick_d_fast

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def nuc_host(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("nuc") / "nuc_host")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_2507_06579_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "nuc_host.cu"), "-o", exe],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("lo,hi", [(10**6, 10**8), (10**10, 10**11), (10**12, 2 * 10**12),
                                   (2**44 - 10**10, 2**44)])
def test_product_lands_on_the_cycle(nuc_host, orc, lo, hi):
    rng = np.random.default_rng(lo % 89 + 3)
    lines, expect = [], []
    for d in _pick_d_fast(orc, rng, lo, hi, 10):
        st = _first_states(d, 1400)  # all inside the first period (_pick_d_fast)
        index = {(Q, P): (j, S, dl) for j, (Q, P, S, dl) in enumerate(st)}
        pairs = [tuple(int(x) for x in rng.integers(0, 500, size=2)) for _ in range(600)]
        pairs += [(5, 5), (40, 40), (0, 0)] + [(i, i + 1) for i in range(20)]
        # the smallest norms of the stretch, against each other and against others
        small = sorted(range(600), key=lambda i: st[i][0])[:12]
        pairs += [(i, k) for i in small for k in small + [100, 200]]
        for i, k in pairs:
            (Qi, Pi, Si, di), (Qk, Pk, Sk, dk) = st[i], st[k]
            lines.append("%d %d %d %d %d %d %d" % (d, Qi // 2, Pi, Si, Qk // 2, Pk, Sk))
            expect.append((d, index, di + dk, math.gcd(Qi // 2, Qk // 2)))
    r = subprocess.run([nuc_host], input="\n".join(lines) + "\n", capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
    rows = r.stdout.strip().split("\n")
    assert len(rows) == len(lines)
    jumped = 0
    for line, (d, index, dsum, common), row in zip(lines, expect, rows):
        st, a, b, g, w, okR, aR, bR, gR = map(int, row.split())
        assert st in (0, 1), line
        if st == 1:
            jumped += common == 1
            continue
        assert common == 1, line
        assert (2 * a, b) in index, line
        j, S, dj = index[(2 * a, b)]
        assert g == S and 4 * a * w == b * b - d, line
        assert abs(dj - dsum) <= math.log(d), line
    assert jumped < 0.02 * len(rows)
