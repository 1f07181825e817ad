"""The cubic-form enumeration at the two ends of wide windows, on the host: every
form that an enumeration in doubles and 128-bit integers finds among the first
and the last candidates is among those the library's job visits, and the forms
decide those candidates as the oracle does.  (A window's ends are where a bound
that is rounded the wrong way loses forms, in a share of the window that does
not shrink with its width.)"""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N = 2000  # candidates looked at, at either end


@pytest.fixture(scope="module")
def wide_host(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("wide") / "cubic_wide_host")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_2507_06579_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "cubic_wide_host.cu"), "-o", exe],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("lo,width", [
    (5, 10**9), (5, 13 * 10**8), (87_941, 2 * 10**9), (930_189, 10**9), (10**9, 10**9),
    (10**9 + 5, 10**10),
    (5, 17 * 10**9),                # the widest single interval of a plan is about this
    (10**11 - 17 * 10**9, 17 * 10**9),
])
def test_no_form_is_lost_at_the_ends(wide_host, orc, lo, width):
    d0 = lo + ((13 - lo % 8) % 8)
    n = (lo + width - d0 + 7) // 8
    for i0 in (0, n - N):
        inp = "".join("%d %d %d %d %d\n" % (d0, n, k, i0, N) for k in (0, 1))
        r = subprocess.run([wide_host], input=inp, capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr
        rows = [ln.split() for ln in r.stdout.strip().split("\n")]
        assert all(int(forms) > N // 10 for _, forms, _ in rows)
        assert [int(lost) for _, _, lost in rows] == [0, 0]
        four, one = (np.frombuffer(row[0].encode(), np.uint8) == ord("1") for row in rows)
        codes = orc.classify_range(d0 + 8 * i0, d0 + 8 * (i0 + N))["codes"]
        assert not np.any(four & (codes == 1))
        assert not np.any((codes == 2) & ~four & ~one)
