"""The fixed-point sums of csrc/soft64.cuh where the operators take over: infinite and NaN values stay what the FP64 sum gives,
sets of subnormal values are not dropped."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2311_04989_gb300", "csrc")


def test_fixed_point_sums_at_the_ends_of_the_range(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text("")
    exe = str(tmp_path / "soft64_edges_host")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(tmp_path), "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "soft64_edges_host.cpp")], check=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split() == ["bad", "0"]
