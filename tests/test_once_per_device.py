"""Shared-memory limits are raised once per device, not once per process: the
class that keeps count on the CPU (tests/once_check.cc), and that every kernel
that needs a limit goes through it."""
import glob
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2502_09541_gb300", "csrc")


def test_once_for_every_device(tmp_path):
    exe = tmp_path / "once_check"
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread", "-I", CSRC, "-o", str(exe),
                           os.path.join(ROOT, "tests", "once_check.cc")])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr


def test_limits_are_raised_in_one_place():
    files = sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*"))
                   if "cudaFuncSetAttribute(" in open(f).read())
    assert files == ["vx_internal.h"]
