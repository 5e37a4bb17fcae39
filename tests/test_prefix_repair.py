"""The repair of a prefix sort on the CPU (tests/prefix_check.cc): groups of one
to twenty pairs with descents everywhere, at the end and nowhere, the bound on a
group's size, stability, and a thread's walk over pair counts up to 2^32 - 1."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_find_and_fix_on_cpu(tmp_path):
    exe = tmp_path / "prefix_check"
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror",
                           "-I", os.path.join(ROOT, "paper_2502_09541_gb300", "csrc"),
                           "-o", str(exe), os.path.join(ROOT, "tests", "prefix_check.cc")])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.endswith("ok\n"), r.stdout + r.stderr
