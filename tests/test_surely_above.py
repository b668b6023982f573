"""The FP32 bound by which gr_con2prim's first pass queues cells (surely_above in csrc/soft64.cuh): it never queues a cell below the
atmosphere threshold, and queues every cell more than its margin above the bound."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2311_04989_gb300", "csrc")


def test_the_bound_is_one_sided_and_fires(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text("")
    exe = str(tmp_path / "surely_above_host")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(tmp_path), "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "surely_above_host.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out[:4] == ["wrong", "0", "missed", "0"] and int(out[5]) > 500000, out
