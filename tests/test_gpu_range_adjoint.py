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
