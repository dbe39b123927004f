"""What the local sum of plans without pair lists keeps of densities far below the largest of their window.

Bar: every product is a float pair, so a sum over old densities alone is as good as any other, up to the
curvature terms' single floats.  Where only the first weights past a kink contribute, those terms are of the
size of the sum: a few 2^-24 of it, 1e-6 with room."""
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


@pytest.mark.parametrize("tol,p", [(1e-12, 8), (1e-6, 4), (1e-14, 16)])
def test_old_densities_of_a_growing_history(tol, p):
    """One driven spring whose density grows by e a step, weak ones at 0.2 to 0.95 of the window's width from
    it: each sees only the densities that are as many steps old, down to e^-45 of the newest."""
    dt, n = 1e-3, 50
    W = int(np.ceil(4 * np.log(1 / tol) / np.pi))
    x = -0.5 + W * dt * np.array([0.0, 0.2, 0.4, 0.6, 0.8, 0.95])
    c = []
    for lw in (0, 1):
        plan = wave1d.Plan(x, np.full(x.size, 1e-8), 1, dt, n, tol, p=p, step_kernel=0, local_weights=lw)
        try:
            for i in range(n):
                g = np.zeros(x.size)
                g[0] = np.exp(i - n)
                plan.step(g)
            c.append(plan.inspect(wave1d.WAVE1D_ARR_LOCAL))
        finally:
            plan.close()
    assert np.all(c[0] != 0.0)
    assert np.max(np.abs(c[1] / c[0] - 1.0)) < 1e-6, c[1] / c[0] - 1.0


@pytest.mark.parametrize("M,span,W,NL", [(1500, 0.03, 0, 0),        # dense: every record is made
                                         (700, 2.0, 0, 0),          # sparse: those that some pair reads
                                         (1600, 0.18, 210, 32),     # dense, a window too long for the copied coefficients
                                         (300, 2.0, 210, 32)])      # sparse, long window
def test_forms_of_the_fold_against_stored_weights(M, span, W, NL):
    """Bar: 1e-10, as everywhere between the two plans (tests/test_gpu_range.py)."""
    rng = np.random.default_rng(M)
    x = np.sort(rng.uniform(-0.5 * span, 0.5 * span, M))
    dt, n = 1e-3, 12
    out = []
    for lw in (0, 1):
        plan = wave1d.Plan(x, np.full(M, 0.2), 0, dt, n, 1e-6, [1.0], [-0.1], [0.3], [-0.3 * span, 0.01],
                           p=4, W=W, NL=NL, local_weights=lw)
        try:
            out.append(plan.solve(n))
        finally:
            plan.close()
    (s0, u0), (s1, u1) = out
    assert np.max(np.abs(s0)) > 1e-3
    assert np.max(np.abs(s1 - s0)) < 1e-10 * np.max(np.abs(s0)) and np.max(np.abs(u1 - u0)) < 1e-10 * np.max(np.abs(u0))
