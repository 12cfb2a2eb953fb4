"""The host's plan of the CTA-pair kernel (tests/pair_plan.cpp): every chunk of T' holds ranks, tiles cover the problem and stay within the
accumulator and the workspace."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_plans(tmp_path):
    exe = str(tmp_path / "pair_plan")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", os.path.join(HERE, "pair_plan.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120).stdout
    assert out == "ok\n", out
