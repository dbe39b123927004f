"""The pair kernels' walk of plans without pair lists, on the CPU (tests/native/pair_walk_check.cpp): every pair closer
than delta is met once whatever the parts, and the sums through it equal the stored FP64 weights'.

Bars, as for the other traversals of the same arithmetic (tests/test_host_range.py): 4e-11 of the largest row sum
(1e-11 where rows hold many pairs), 1e-9 for the transposed sums."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_host_range import CSRC, HERE, INCLUDE, _layout


@pytest.fixture(scope="module")
def checker():
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    build_dir = os.path.join(HERE, "native", "_build")
    os.makedirs(build_dir, exist_ok=True)
    out = os.path.join(build_dir, "pair_walk_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-I", INCLUDE, "-o", out,
                    os.path.join(HERE, "native", "pair_walk_check.cpp"), os.path.join(CSRC, "plan_host.cpp"), "-lpthread"],
                   check=True, capture_output=True)
    return out


@pytest.mark.parametrize("part", [0, 16])
@pytest.mark.parametrize("name,bar", [("uniform", 4e-11), ("cluster", 1e-11), ("seam", 4e-11), ("coincident", 4e-11),
                                      ("single", 4e-11), ("grouped", 1e-11), ("sparse", 4e-11)])
def test_every_pair_once_and_the_stored_weights_sums(checker, name, bar, part):
    bc, dt, tol, x = _layout(name, np.random.default_rng(9))
    x = x[:1200]
    text = f"{x.size} {dt!r} {tol!r} {bc} {part}\n" + " ".join(repr(float(v)) for v in x) + "\n"
    r = subprocess.run([checker], input=text, capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
    wrong, err, terr, pairs = r.stdout.split()[1:]
    assert int(wrong) == 0 and int(pairs) >= x.size
    assert float(err) < bar and float(terr) < 1e-9, (err, terr)


def test_tables_do_not_depend_on_the_environment(checker):
    bc, dt, tol, x = _layout("coincident", np.random.default_rng(9))
    text = f"{x.size} {dt!r} {tol!r} {bc} 0\n" + " ".join(repr(float(v)) for v in x) + "\n"
    out = [subprocess.run([checker], input=text, capture_output=True, text=True, env=env).stdout
           for env in (os.environ, dict(os.environ, WAVE1D_RANGE_WIDTH="0.45"))]
    assert out[0].startswith("ok") and out[0] == out[1]
