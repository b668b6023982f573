"""The FP32 conversions of a mixed stage (csrc/castlist.h): the list holds every pool of the fullest stage (table EOS,
extrinsic curvature, no FP32 copies from the caller: 25), with each pool's own destination and length."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

# what the header needs of the CUDA headers on a host without them
STUB = """#pragma once
#include <cstdint>
#define __host__
#define __device__
#define __forceinline__ inline
struct int2 { int x, y; };
struct int4 { int x, y, z, w; };
typedef int cudaError_t;
typedef void* cudaStream_t;
typedef void* cudaEvent_t;
"""


def test_cast_list_holds_every_pool_of_the_fullest_stage(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(STUB)
    exe = str(tmp_path / "castlist_host")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Wno-unused-function", "-I", str(tmp_path), "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2311_04989_gb300", "csrc"), "-o", exe,
                    os.path.join(HERE, "castlist_host.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out[:2] == ["bad", "0"], out
    assert int(out[3]) == 25 and int(out[5]) >= 25, out
