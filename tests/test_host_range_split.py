"""The cut of the distance intervals of a plan without pair lists, on the CPU: parts (they set the order of the
local sum) follow from the layout alone, slabs (memory) are whole parts whatever memory is free."""
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
    build_dir = os.path.join(HERE, "native", "_build")
    os.makedirs(build_dir, exist_ok=True)
    out = os.path.join(build_dir, "range_split_check")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", INCLUDE, "-o", out, os.path.join(HERE, "native", "range_split_check.cpp"),
                    os.path.join(CSRC, "plan_host.cpp"), "-lpthread"], check=True, capture_output=True)
    return out


@pytest.mark.parametrize("nint,M,pairs", [(3, 1, 1), (21, 40, 100), (484, 3000, 250_000), (676, 16_383, 4_000_000), (676, 16_384, 4_000_000),
                                          (676, 100_000, 153_000_000), (484, 1_000_000, 13_400_000_000), (32_767, 50_000, 10**9),
                                          (676, 10_000_000, 10**12), (676, 500_000_000, 10**15)])
def test_parts_do_not_depend_on_free_memory(checker, nint, M, pairs):
    r = subprocess.run([checker], input=f"{nint} {M} {pairs}\n", capture_output=True, text=True, check=True)
    rows = [list(map(int, line.split())) for line in r.stdout.splitlines()]
    parts = {(part, nparts) for _, part, nparts, _ in rows}
    assert len(parts) == 1, rows
    (part, nparts), = parts
    assert part % 16 == 0 and part >= 16 and part * nparts >= nint > part * (nparts - 1)
    slabs = [slab for *_, slab in rows]
    assert all(s >= part and s % part == 0 for s in slabs) and slabs == sorted(slabs, reverse=True) and slabs[-1] == part
    # with memory to spare: 16 KB a spring (8 KB below 16384), 4 GiB, no more than the intervals
    most = max(16, min((nint + 15) // 16 * 16, min((8192 if M < 16384 else 16384) * M, 4 << 30) // (48 * M) // 16 * 16))
    assert slabs[0] == most // part * part
