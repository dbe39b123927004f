"""Sizes at the edges of the kernels' tiles: rows and springs of the local sum, the implicit sweeps and
the receivers of plans without pair lists (tiles of 8, 16, 64 and 128 springs, the sweeps' cluster of 8
blocks up to 8192 springs and of 16 above), and the segments of 64 points of the FP64 spreading.

Bars: the range tables hold every weight to 1e-12 of max |Q|, single-float curvature terms make that 2e-11
of a row's sum where rows hold few sources: 1e-10 against the stored-weight plan.  FP64 NUFFT at tol 1e-12:
1e-10 of the largest direct sum."""
import numpy as np
import pytest

from oracle import wfp
from paper_2507_07823_gb300 import build, wave1d
from paper_2507_07823_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    wave1d.lib()


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


@pytest.mark.parametrize("M", [1, 15, 33, 127, 129, 1025, 8192, 8193, 12001])
def test_range_plan_at_tile_edges(M):
    """Springs under the pulse from the first step on, 0.6 per dt at the largest size."""
    rng = np.random.default_rng(100 + M)
    dt = 1e-3 if M < 2000 else 3e-4
    x = np.sort(rng.uniform(-np.pi, np.pi, M)) if M > 1 else np.array([-1.95])
    w = W.make(M=M, bc=W.PERIODIC, dt=dt, Nt=40, tol=1e-10, p=4, seed=M, R=4)
    w = w.with_(x=x, beta=rng.uniform(1.0, 10.0, M), xr=np.array([-2.05, -1.9, x[0], 3.0]))
    out = []
    for lw in (0, 1):
        plan = wave1d.Plan.from_workload(w, local_weights=lw)
        try:
            out.append(plan.solve(w.Nt))
        finally:
            plan.close()
    (s0, u0), (s1, u1) = out
    assert np.max(np.abs(s0)) > 1e-3
    assert _rel(s1, s0) < 1e-10 and _rel(u1, u0) < 1e-10, (_rel(s1, s0), _rel(u1, u0))


@pytest.mark.parametrize("M", [1, 2, 63, 64, 65, 129, 4097])
@pytest.mark.parametrize("layout", ["uniform", "one_cell"])
def test_fp64_spreading_segments(M, layout):
    """Points over the whole period, and all but the last of them in one cell beside the seam."""
    K = 315
    rng = np.random.default_rng(M)
    x = rng.uniform(-np.pi, np.pi, M)
    if layout == "one_cell":
        x[: M - 1] = np.pi - 1e-9 * rng.uniform(1.0, 2.0, M - 1)
    c = rng.uniform(0.5, 1.5, M)
    alpha = rng.standard_normal(K + 1) + 1j * rng.standard_normal(K + 1)
    alpha[0] = alpha[0].real
    import torch
    nu = wave1d.Nufft(x, K, 1e-12, 0)
    try:
        cd = torch.tensor(c[nu.perm], device="cuda")
        Sd = torch.zeros(2 * (K + 1), dtype=torch.float64, device="cuda")
        ad = torch.tensor(np.stack([alpha.real, alpha.imag], 1).reshape(-1), device="cuda")
        ud = torch.zeros(M, dtype=torch.float64, device="cuda")
        nu.type1(cd, Sd)
        nu.type2(ad, ud)
        torch.cuda.synchronize()
        S, u = Sd.cpu().numpy(), np.empty(M)
        u[nu.perm] = ud.cpu().numpy()
    finally:
        nu.close()
    assert _rel(S[0::2] + 1j * S[1::2], wfp.type1(c, x, K)) < 1e-10
    assert np.max(np.abs(u - wfp.type2(alpha, x))) < 1e-10 * np.sum(np.abs(alpha))
