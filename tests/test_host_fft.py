"""The complex transforms behind the exact products of encryption and decryption, compiled for
the CPU and run thread by thread: index arithmetic, tables and the rounding-error bounds; and what a kernel does when a copy does not come."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("logn", [0, 13, 14, 15, 16])
def test_exact_products_on_the_host(tmp_path, logn):
    exe = str(tmp_path / "host_fft_check")
    cmd = ["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-o", exe,
           os.path.join(ROOT, "tests", "host_fft_check.cpp"),
           os.path.join(ROOT, "paper_2303_10837_b200", "csrc", "fedhe_host.cpp"), "-lquadmath"]
    build = subprocess.run(cmd, capture_output=True, text=True)
    assert build.returncode == 0, build.stderr[-4000:]
    run = subprocess.run([exe, str(logn)], capture_output=True, text=True, timeout=600)
    assert run.returncode == 0 and run.stdout.strip().endswith("ok"), run.stdout[-2000:] + run.stderr[-2000:]
