"""How the thread blocks of a sequence settle its status word (csrc/seq_status.cuh), in every order of their steps, on the CPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_order_of_the_blocks_steps_loses_a_failure(tmp_path):
    exe = str(tmp_path / "orders")
    subprocess.run(["g++", "-std=c++17", "-O2", "-x", "c++", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2408_00264_b200", "csrc"),
                    os.path.join(ROOT, "tests", "seq_status_orders.cpp"), "-o", exe], check=True, timeout=120)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 10000
