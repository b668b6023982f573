"""The integer forms of FP64 operations (csrc/soft64.cuh) against the IEEE operations of the host: division, square
root, the difference of two FP32 values, widening and comparisons bit for bit, the reciprocal square root within 0.65
ulp (its stated bound), the eight-value mean within one rounding and 2^-58 of the largest addend."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2311_04989_gb300", "csrc")


def test_integer_fp64_operations_match_ieee(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text("")   # the header needs nothing of it on the host
    exe = str(tmp_path / "soft64_host")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(tmp_path), "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "soft64_host.cpp")], check=True)
    out = subprocess.run([exe, "4000000"], check=True, capture_output=True, text=True).stdout.split()
    assert out[0] == "bad" and int(out[1]) == 0, out
    assert float(out[3]) <= 0.65, out
