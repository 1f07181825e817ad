"""The cubic-form enumeration on the host under the compiler's check for signed
overflow (an overflow ends the program)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_signed_overflow(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "cubic_host")
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-Xcompiler", "-fsanitize=signed-integer-overflow",
                        "-Xcompiler", "-fno-sanitize-recover=all",
                        "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_2507_06579_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "cubic_host.cu"), "-o", exe, "-lubsan"],
                       capture_output=True, text=True, timeout=300)
    if r.returncode != 0 and "ubsan" in r.stderr:
        pytest.skip("no libubsan")
    assert r.returncode == 0, r.stderr
    windows = [(5, 1), (5, 20_000), (10**9 + 5, 3_000), (10**11 - 99_987 * 10, 500)]
    inp = "".join("%d %d %d\n" % (d0 + (13 - d0 % 8) % 8, n, k) for d0, n in windows for k in (0, 1))
    r = subprocess.run([exe], input=inp, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert len(r.stdout.strip().split("\n")) == 2 * len(windows)
