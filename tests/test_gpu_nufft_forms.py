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
