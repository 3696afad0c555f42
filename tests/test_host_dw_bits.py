"""The integer conversions between FP64 and double words (csrc/dw.cuh), compiled for
the host: the split equals the rounded conversions bit for bit, the recombination
rounds to nearest, and zeros, infinities and NaN keep their meaning (CPU)."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def test_conversions_bit_exact(tmp_path):
    if not os.path.isdir(os.path.join(CUDA, "include")):
        pytest.skip("no CUDA headers")
    exe = str(tmp_path / "dw_bits")
    src = os.path.join(HERE, "host", "dw_bits.cpp")
    inc = os.path.join(HERE, "..", "paper_2205_11990_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", inc, "-isystem", os.path.join(CUDA, "include"), src,
                    "-o", exe], check=True)
    bad_from, bad_to, edges = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert bad_from == 0 and bad_to == 0 and edges == 1
