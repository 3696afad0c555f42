"""The split of an FP64 value into a double word (csrc/dw.cuh), compiled for the host,
keeps both words of values far below their scale as long as FP32 has them (CPU)."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def test_small_values_keep_both_words(tmp_path):
    if not os.path.isdir(os.path.join(CUDA, "include")):
        pytest.skip("no CUDA headers")
    exe = str(tmp_path / "dw_small")
    inc = os.path.join(HERE, "..", "paper_2205_11990_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", inc, "-isystem", os.path.join(CUDA, "include"),
                    os.path.join(HERE, "host", "dw_small.cpp"), "-o", exe], check=True)
    assert int(subprocess.run([exe], check=True, capture_output=True, text=True).stdout) == 0
