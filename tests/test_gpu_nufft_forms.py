"""Forms of the standalone NUFFTs beside the ones tests/test_gpu_nufft.py compares with direct sums."""
import numpy as np
import pytest

from paper_2507_07823_gb300 import build, wave1d

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    wave1d.lib()


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-6)])
@pytest.mark.parametrize("instances", [1, 3])
def test_arrays_at_odd_offsets(precision, tol, instances):
    """Every array is aligned to a double and no more (the k-th value of a larger buffer): the same bits as
    from 16-byte aligned arrays, and nothing beside the arrays is written."""
    import torch
    rng = np.random.default_rng(8)
    sets = [rng.uniform(-np.pi, np.pi, m) for m in (37, 2500, 640)[:instances]]
    K = 300
    nu = wave1d.Nufft(sets if instances > 1 else sets[0], K, tol, precision)
    try:
        sizes = dict(c=nu.M, S=instances * 2 * (K + 1), a=instances * 2 * (K + 1), u=nu.M)
        even = {k: torch.from_numpy(rng.standard_normal(n)).cuda() for k, n in sizes.items()}
        bufs = {k: torch.full((n + 2,), -7.0, dtype=torch.float64, device="cuda") for k, n in sizes.items()}
        odd = {k: bufs[k][1:-1] for k in sizes}
        assert all(v.data_ptr() % 16 == 8 for v in odd.values()) and all(v.data_ptr() % 16 == 0 for v in even.values())
        for k in ("c", "a"):
            odd[k].copy_(even[k])
        for v in (even, odd):
            nu.type1(v["c"], v["S"])
            nu.type2(v["a"], v["u"])
        torch.cuda.synchronize()
        assert torch.equal(even["S"], odd["S"]) and torch.equal(even["u"], odd["u"])
        assert all(float(b[0]) == -7.0 and float(b[-1]) == -7.0 for b in bufs.values())
    finally:
        nu.close()


@pytest.mark.parametrize("precision,tol,rel", [(0, 1e-10, 1e-12), (1, 1e-6, 1e-6)])
def test_autotuner_cuts_what_the_spreading_runs(precision, tol, rel):
    """Its caps are those of the spreading in use (FP64: one cell, points of a segment), the spread through them is the
    default split's to rounding, and the tables of the candidates that lost are given back."""
    import torch
    rng = np.random.default_rng(3)
    x = np.concatenate([1.234 + 1e-9 * rng.standard_normal(6000), rng.uniform(-np.pi, np.pi, 500_000)])
    nu = wave1d.Nufft(x, 6283, tol, precision)
    try:
        c = torch.from_numpy(rng.standard_normal(nu.M)).cuda()
        grids = [torch.zeros(nu.nf, dtype=torch.float64, device="cuda") for _ in range(2)]
        nu.spread(c, grids[0])
        caps = {nu.autotune(c, grids[1], reps=2)}
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        for _ in range(6):
            caps.add(nu.autotune(c, grids[1], reps=2))
            nu.spread(c, grids[1])
            assert float((grids[1] - grids[0]).abs().max()) <= rel * float(grids[0].abs().max())
        torch.cuda.synchronize()
        assert abs(torch.cuda.mem_get_info()[0] - free) <= 8 << 20
        assert all((cells == 1 and points in (16, 32, 64, 128, 256)) if precision == 0 else
                   (cells in (60, 120, 240) and points in (512, 1024, 2048)) for cells, points in caps), caps
    finally:
        nu.close()


def test_more_instances_than_one_group_of_ffts():
    """1100 instances at K = 6283: the FFT passes take them in two groups (1024 fine grids of 32768 to a group).  The
    instances beside the cut and at the ends against direct sums."""
    import torch
    from oracle import wfp
    rng = np.random.default_rng(21)
    K, n = 6283, 1100
    sets = [rng.uniform(-np.pi, np.pi, 1 + i % 4) for i in range(n)]
    nu = wave1d.Nufft(sets, K, 1e-10, 0)
    try:
        assert nu.nf == 32768
        c = rng.standard_normal(nu.M)
        a = rng.standard_normal((n, K + 1, 2))
        a[:, 0, 1] = 0.0
        S = torch.zeros(n, K + 1, 2, dtype=torch.float64, device="cuda")
        ud = torch.zeros(nu.M, dtype=torch.float64, device="cuda")
        nu.type1(torch.from_numpy(c[nu.perm]).cuda(), S)
        nu.type2(torch.from_numpy(a).cuda(), ud)
        u = np.empty(nu.M)
        u[nu.perm] = ud.cpu().numpy()
        off = nu.offsets
        for i in (0, 511, 1022, 1023, 1024, 1025, n - 1):
            ref = wfp.type1(c[off[i]:off[i + 1]], sets[i], K)
            got = S[i].cpu().numpy() @ np.array([1.0, 1j])
            assert np.max(np.abs(got - ref)) < 1e-8 * np.max(np.abs(ref))
            ref = wfp.type2(a[i] @ np.array([1.0, 1j]), sets[i])
            assert np.max(np.abs(u[off[i]:off[i + 1]] - ref)) < 1e-8 * np.sum(np.abs(a[i]))
    finally:
        nu.close()
