"""The recorded steps of a quadratic run for lists in any order, on the CPU: the
kernels' loop over them ends whatever the list holds (tests/records_check.cpp
compiles its logic from the library's own header)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_30342_gb300", "csrc")


def test_every_list_ends_and_records_the_right_steps(tmp_path):
    exe = tmp_path / "records_check"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, os.path.join(ROOT, "tests", "records_check.cpp"),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip().endswith("OK"), out.stdout + out.stderr
