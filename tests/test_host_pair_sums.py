"""Sums of float pairs that stand where FP64 sums stood (range.cuh, acc3_add), on the CPU.

The sum is exact but for the two roundings to a double of the harness (one where it is carried from slab to
slab, one at the end): 2 x 2^-53 of the terms' magnitudes, far below it where they cancel.  Kept as one pair it
loses 2^-24 of its low part at each addition."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2507_07823_gb300", "csrc")


def test_sums_in_three_floats_are_as_good_as_fp64():
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    build_dir = os.path.join(HERE, "native", "_build")
    os.makedirs(build_dir, exist_ok=True)
    out = os.path.join(build_dir, "pair_sums_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-o", out,
                    os.path.join(HERE, "native", "pair_sums_check.cpp")], check=True, capture_output=True)
    r = subprocess.run([out], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
    three, one = map(float, r.stdout.split()[1:])
    assert three <= 2.0 < one, (three, one)
