"""The plan of the persistent launches (csrc/ca_steps_plan.h), compiled for the host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_steps_plan(tmp_path):
    exe = tmp_path / "steps_plan_check"
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror",
                    "-I" + os.path.join(ROOT, "paper_1612_04003_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "steps_plan_check.cpp"), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and "ALL OK" in r.stdout, r.stdout + r.stderr
