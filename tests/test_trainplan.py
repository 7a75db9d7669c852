"""How a mini-batch's pairs are shared out to training lanes (csrc/trainplan.h):
the sums that make up the gradient, and their order, do not depend on how many
lanes the device has memory for."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sums_do_not_depend_on_the_lanes(tmp_path):
    exe = tmp_path / "trainplan_check"
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_1107_0538_gb300", "csrc"),
                    "-o", str(exe), os.path.join(ROOT, "tests", "trainplan_check.cpp")], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
