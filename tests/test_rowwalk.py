"""The row walk of cg_solve_noalloc's products (csrc/rowwalk.h) on the CPU:
every entry once, and no arithmetic past the range of an int at the largest
row pointers (cg_solve_noalloc takes up to 2^31 - 1 entries)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_walks_visit_every_entry_once(tmp_path):
    exe = tmp_path / "rowwalk_check"
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                    "-I", os.path.join(ROOT, "paper_1107_0538_gb300", "csrc"), "-o", str(exe),
                    os.path.join(ROOT, "tests", "rowwalk_check.cpp")], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout + res.stderr
