"""The parts that the reverse march's kernels split an element's work into, added up on the CPU against the plain forms
that tests/test_host_adjoint.py holds to the adjoint oracle: bit for bit where the order of sums is the same, else within
the rounding of a sum of at most 849 terms in another order (1e-13 of the largest value)."""
import os
import shutil
import subprocess

import pytest

from test_host_range import CSRC, HERE, INCLUDE


def test_parts_add_up_to_the_plain_forms():
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    build_dir = os.path.join(HERE, "native", "_build")
    os.makedirs(build_dir, exist_ok=True)
    out = os.path.join(build_dir, "adjoint_parts_check")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-I", INCLUDE, "-o", out,
                    os.path.join(HERE, "native", "adjoint_parts_check.cpp")], check=True, capture_output=True)
    r = subprocess.run([out], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), (r.returncode, r.stdout, r.stderr)
    assert float(r.stdout.split()[1]) < 1e-13
