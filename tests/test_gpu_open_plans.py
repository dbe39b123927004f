"""Plans open beside one another: opening a smaller plan changes nothing for a larger one that is open already."""
import numpy as np
import pytest

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


def _workload(dt, tol):
    rng = np.random.default_rng(12)
    return W.Workload(name="open", bc=W.PERIODIC, x=np.sort(rng.uniform(-3.0, 3.0, 300)), beta=rng.uniform(1.0, 5.0, 300),
                      amp=np.array([1.0]), center=np.array([-1.0]), width=np.array([0.5]), dt=dt, Nt=40, tol=tol, p=4,
                      xr=np.array([-1.0, 0.5]), seed=12)


@pytest.mark.parametrize("opt", [{}, {"step_kernel": 0}, {"local_weights": 1}, {"local_weights": 1, "precision": 1}])
def test_a_smaller_plan_opened_later_leaves_the_larger_one_alone(opt):
    """Modes 6283 against 157, windows of 18 against 9 steps (the kernels' shared memory follows both), single
    steps with a forcing vector and the captured march: the same bits with and without the second plan."""
    large, small = _workload(5e-4, 1e-6), _workload(0.02, 1e-3)
    g = np.linspace(0.1, 1.0, large.M)
    out = []
    for second in (False, True):
        plan = wave1d.Plan.from_workload(large, **opt)
        other = wave1d.Plan.from_workload(small, **opt) if second else None
        try:
            plan.step(g)
            out.append((plan.sigma(), *plan.solve(large.Nt - 1)))
            if other:
                other.solve(small.Nt)
        finally:
            plan.close()
            if other:
                other.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("opt", [{}, {"step_kernel": 0}])
def test_a_smaller_batch_opened_later_leaves_the_larger_one_alone(opt):
    out = []
    for second in (False, True):
        batch = wave1d.Batch([_workload(5e-4, 1e-10)] * 2, **opt)
        other = wave1d.Batch([_workload(0.02, 1e-10)], **opt) if second else None
        try:
            out.append(batch.solve(40))
        finally:
            batch.close()
            if other:
                other.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
