"""Error samplers: the tables that decide a sample by its high word, on the host, against the thresholds themselves."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sampler_tables_on_the_host(tmp_path):
    exe = str(tmp_path / "host_gauss_check")
    build = subprocess.run(["g++", "-O2", "-std=gnu++17", "-o", exe, os.path.join(ROOT, "tests", "host_gauss_check.cpp")],
                           capture_output=True, text=True)
    assert build.returncode == 0, build.stderr[-4000:]
    run = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert run.returncode == 0, run.stdout[-2000:] + run.stderr[-2000:]
