"""The lane search as its kernels run it (nuc_stride, nuc_mul cycles with steps
where norms share a factor, the filter), modelled on the host: every hit lies at
l - j or l + j of the first period with the oracle's class, the filter holds
every entry, and the steps that come out of the window's margin keep to their
bounds."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_bsgs_host import _ds

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def stride_host(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("stride") / "stride_host")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_2507_06579_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "stride_host.cu"), "-o", exe],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return exe


def _run(exe, rows):
    r = subprocess.run([exe], input="".join("%d %d %d %d\n" % x for x in rows), capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stderr
    out = [tuple(int(x) for x in ln.split()) for ln in r.stdout.strip().split("\n")]
    assert len(out) == len(rows)
    return out


@pytest.mark.parametrize("lo,hi,n,settings,verify", [
    (10**8, 10**9, 150, ((300, 8), (640, 16)), 1),
    (10**9, 10**10, 150, ((300, 8), (640, 16), (1200, 32)), 1),
    (10**11 - 10**9, 10**11, 40, ((768, 14), (1024, 16)), 0),
    (2**44 - 10**9, 2**44, 12, ((2048, 28), (4096, 51)), 0),
])
def test_every_hit_is_in_the_first_period(stride_host, orc, lo, hi, n, settings, verify):
    rng = np.random.default_rng(lo % 101)
    rows = [(d, N, m, verify) for d in _ds(orc, rng, lo, hi, n) for N, m in settings]
    searched = 0
    for (d, N, m, _), (status, g, cycles, steps, stride, filtered, hit) in zip(rows, _run(stride_host, rows)):
        assert status in (0, 1, 2), (d, N, m, status)
        assert filtered == 0 and steps <= 32 and stride <= 24
        if status < 2:
            rc, theta, _ = orc.walk_mod2(d)
            assert rc == 0 and g == theta - 1, (d, N, m)
        if status == 1:
            searched += 1
            assert hit == verify, (d, N, m)
    assert searched > len(rows) // 2


def test_strides_from_any_two_states_keep_to_their_steps(stride_host, orc):
    """Every pair of marked states (the smallest norms share factors most often):
    on the cycle with the right class and coefficient, within 24 steps."""
    rng = np.random.default_rng(5)
    rows = [(d, 2000, 16, 2) for d in _ds(orc, rng, 10**10, 10**11, 25)]
    out = _run(stride_host, rows)
    assert sum(o[1] for o in out) > 10**5
    assert all(o[4] == 0 and o[3] <= 24 for o in out)
    assert sum(o[2] for o in out) > 0.999 * sum(o[1] for o in out)
    assert max(o[3] for o in out) > 16  # the bound is met
