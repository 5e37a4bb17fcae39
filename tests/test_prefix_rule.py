"""Which inputs of a pair sort go to the prefix sort, on the CPU
(tests/prefix_rule_check.cc): keys that occur once or twice do, keys that occur
ten times or more, whose prefix groups are too large to repair, do not."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_repeating_keys(tmp_path):
    exe = tmp_path / "prefix_rule_check"
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-Wall", "-Werror",
                           "-I", os.path.join(ROOT, "paper_2502_09541_gb300", "csrc"),
                           "-o", str(exe), os.path.join(ROOT, "tests", "prefix_rule_check.cc")])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr
