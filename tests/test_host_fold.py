"""The operands of the tensor-core fold of plans without pair lists (opts.local_weights = 1), on the CPU.

tests/native/fold_check.cpp contracts the plan builder's coefficient slices with the density slices of
csrc/range.cuh as the kernel does and compares every power's sum with FP64.  Bounds, from the slices: e_0 drops
products below 2^-43 of the largest |a sigma| of up to 4 accumulations of m_max terms, and the higher powers'
coefficients are smaller by more than the slices they lack, so 41 terms x 4 x 2^-44 = 1e-11 bounds the worst case and
1e-12 the sums of terms of random sign checked here.  Partial sums must stay whole numbers of FP32, below 2^24.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2507_07823_gb300", "csrc")
INCLUDE = os.path.join(HERE, "..", "include")


@pytest.fixture(scope="module")
def checker():
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    build_dir = os.path.join(HERE, "native", "_build")         # git-ignored, inside the repository
    os.makedirs(build_dir, exist_ok=True)
    out = os.path.join(build_dir, "fold_check")
    cmd = ["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-I", INCLUDE, "-o", out,
           os.path.join(HERE, "native", "fold_check.cpp"), os.path.join(CSRC, "plan_host.cpp"), "-lpthread"]
    subprocess.run(cmd, check=True, capture_output=True)
    return out


@pytest.mark.parametrize("dt,tol,p", [(5e-4, 1e-10, 4), (1e-3, 1e-12, 8), (5e-4, 1e-6, 4), (1e-3, 1e-8, 6), (0.01, 1e-13, 16), (0.02, 1e-3, 2)])
@pytest.mark.parametrize("spread", [0.0, 12.0])
def test_slices_carry_the_fold(checker, dt, tol, p, spread):
    r = subprocess.run([checker], input=f"{dt!r} {tol!r} {p} {spread!r}\n", capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
    _, err, most = r.stdout.split()
    assert float(err) < 1e-12, err
    assert float(most) < 2 ** 24, most
