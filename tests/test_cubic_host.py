"""The cubic-form enumeration (eis_cubic.cuh), run on the host against the
oracle: over every candidate of a window, a form of discriminant 4d means
d in E, and a square-free d with neither a form of discriminant 4d nor one of
discriminant d is not in E (so every d in E has one or the other)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def cubic_host(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("cubic") / "cubic_host")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_2507_06579_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "cubic_host.cu"), "-o", exe],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("lo,n", [
    (5, 1), (5, 2), (37, 1),                # the smallest discriminants, one candidate
    (5, 125_000),                           # the small configuration, from the bottom
    (10**7 + 3, 20_011), (4 * 10**8, 10_000), (10**9, 30_000),
    (10**11 - 10**5, 4_000),                # the benchmark's decade
    (10**12 - 8 * 700, 700),
])
def test_forms_decide_as_the_oracle(cubic_host, orc, lo, n):
    d0 = lo + ((13 - lo % 8) % 8)
    r = subprocess.run([cubic_host], input="%d %d 0\n%d %d 1\n" % (d0, n, d0, n),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0
    four, one = (np.frombuffer(ln.split()[0].encode(), np.uint8) == ord("1")
                 for ln in r.stdout.strip().split("\n"))
    codes = orc.classify_range(d0, d0 + 8 * n)["codes"]
    assert len(codes) == len(four) == len(one) == n
    sqfree, in_e = codes > 0, codes == 2
    assert not np.any(four & sqfree & ~in_e)
    assert not np.any(in_e & ~four & ~one)
    if n >= 10_000:  # they decide most d: the undecided are about a tenth
        assert (sqfree & one & ~four).sum() < 0.16 * sqfree.sum()
