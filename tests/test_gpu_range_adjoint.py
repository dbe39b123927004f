"""Reverse march of plans without pair lists against the stored-weight plan of the same layout, on the same
densities: window lengths from one group of steps of the transposed local sum's kernel to several.

Bar: 1e-9 of the largest component, the bar between the two forms (the curvature moments are single floats)."""
import numpy as np
import pytest

from paper_2507_07823_gb300 import build, wave1d
from paper_2507_07823_gb300 import workloads as W

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    wave1d.lib()


@pytest.mark.parametrize("bc", [W.PERIODIC, W.FREE])
@pytest.mark.parametrize("M,tol,p,opt", [(1, 1e-10, 4, {}), (65, 1e-3, 2, {}), (300, 1e-12, 8, {}), (1100, 1e-13, 16, {}),
                                         (130, 1e-6, 4, dict(W=70, NL=32)), (150, 1e-6, 4, dict(W=210, NL=32))])
def test_gradients_match_the_stored_weight_plan(bc, M, tol, p, opt):
    rng = np.random.default_rng(M)
    x = np.sort(rng.uniform(-0.4, 0.4, M))
    w = W.Workload(name="adjoint", bc=bc, x=x, beta=rng.uniform(0.5, 2.0, M), amp=np.array([1.0]), center=np.array([-0.2]),
                   width=np.array([0.3]), dt=1e-3, Nt=60, tol=tol, p=p, xr=np.array([-0.5, x[M // 2], 0.45]), seed=M)
    ubar = torch.from_numpy(rng.standard_normal((w.Nt, 3))).cuda()
    sigma, out = None, []
    for lw in (0, 1):
        plan = wave1d.Plan.from_workload(w, local_weights=lw, **opt)
        try:
            if sigma is None:
                sigma, _ = plan.solve_device(w.Nt)
            out.append([v.cpu().numpy() for v in plan.adjoint(sigma, ubar, forcing_gradient=True)])
        finally:
            plan.close()
    for a, b in zip(*out):
        assert np.max(np.abs(a)) > 0 and np.max(np.abs(b - a)) <= 1e-9 * np.max(np.abs(a))


def test_reverse_march_of_a_mixed_plan():
    """Mixed plans march back in FP64 through the same kernels: the gradients of the FP64 plan without pair lists from
    the same densities (bar: 1e-10, the sweeps' stopping rule and order), the same bits from call to call, and no
    memory kept by the plan; from checkpoints the same bits as from stored densities."""
    rng = np.random.default_rng(5)
    M = 900
    x = np.sort(rng.uniform(-0.6, 0.6, M))
    w = W.Workload(name="mixed", bc=W.FREE, x=x, beta=rng.uniform(0.5, 2.0, M), amp=np.array([1.0]), center=np.array([-0.2]),
                   width=np.array([0.3]), dt=1e-3, Nt=40, tol=1e-6, p=4, xr=np.array([-0.7, x[11], 0.65]), seed=5)
    ubar = torch.from_numpy(rng.standard_normal((w.Nt, 3))).cuda()
    f64 = wave1d.Plan.from_workload(w, local_weights=1)
    mixed = wave1d.Plan.from_workload(w, local_weights=1, precision=1)
    ck = wave1d.Plan.from_workload(w, local_weights=1, precision=1)
    try:
        sigma, _ = mixed.solve_device(w.Nt)
        a = f64.adjoint(sigma, ubar, forcing_gradient=True)
        before = wave1d.wave1d_get_info(mixed.h).device_bytes
        b = mixed.adjoint(sigma, ubar, forcing_gradient=True)
        c = mixed.adjoint(sigma, ubar, forcing_gradient=True)
        assert wave1d.wave1d_get_info(mixed.h).device_bytes == before
        _, buf = ck.solve_checkpointed(w.Nt, 7)
        d = ck.adjoint_checkpointed(buf, w.Nt, 7, ubar, forcing_gradient=True)
        for u, v, s, t in zip(a, b, c, d):
            assert float((v - u).abs().max()) <= 1e-10 * float(u.abs().max()) and float(u.abs().max()) > 0
            assert torch.equal(v, s) and torch.equal(v, t)
    finally:
        for plan in (f64, mixed, ck):
            plan.close()


@pytest.mark.parametrize("lw", [0, 1])
def test_more_receivers_than_the_table_of_waves_holds(lw):
    """1400 receivers at 3142 modes pass the 64 MB of the receivers' waves, which are then formed at each step: the
    gradient is the sum of those of the two halves of the receivers (bar: 1e-12, the order of the sums)."""
    rng = np.random.default_rng(2)
    M, n, R = 40, 20, 1400
    xr = np.sort(rng.uniform(-1.0, 1.0, R))
    ubar = torch.from_numpy(rng.standard_normal((n, R))).cuda()
    w = W.Workload(name="waves", bc=W.FREE, x=np.sort(rng.uniform(-0.5, 0.5, M)), beta=rng.uniform(0.5, 2.0, M), amp=np.array([1.0]),
                   center=np.array([-0.2]), width=np.array([0.3]), dt=1e-3, Nt=n, tol=1e-8, p=4, xr=xr, seed=2)
    out, sigma = [], None
    for part in (slice(0, R), slice(0, R // 2), slice(R // 2, R)):
        plan = wave1d.Plan.from_workload(w.with_(xr=xr[part]), local_weights=lw)
        try:
            if sigma is None:
                sigma, _ = plan.solve_device(n)
            out.append(plan.adjoint(sigma, ubar[:, part].contiguous(), forcing_gradient=True))
        finally:
            plan.close()
    for whole, a, b in zip(*out):
        assert float((a + b - whole).abs().max()) <= 1e-12 * max(float(a.abs().max()), float(b.abs().max()))
