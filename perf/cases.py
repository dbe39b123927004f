"""What a user of this framework has it do, as cases to be timed: marches of point springs in the periodic box and
in free space, single driven steps, gradients by the reverse march, batches of instances, and the history part's
NUFFTs alone.  Sizes are those of `workloads.py` (the paper's experiments and the configurations beside them), of the
tests and of the benchmark, with odd ones between them.

Every march starts from rest and is driven by pulses that lie over the springs, so that every density and receiver is
live from the first step (the paper's disordered medium keeps its own pulse, which has run into it by then).
`prepare` marches on until the window of W steps is full of history, or well into it where a step is dear: a pass
is a few steps of a march under way.
"""
import math

import numpy as np
import torch

from paper_2507_07823_gb300 import wave1d, workloads

BOX, FREE = workloads.PERIODIC, workloads.FREE


def listed():
    return [
        # the smallest plan (periodic box, 64 springs): a step is latency and launches
        dict(name="box_64", kind="march", bc=BOX, M=64, layout="uniform", dt=0.01, tol=1e-10, p=8, R=4, steps=64, lead=64),
        # the paper's disordered medium with its space-time readout: 150 springs, 100 receivers, one
        # radiation projection in each pass
        dict(name="media_150", kind="media", beta_max=5.0, steps=54, lead=162),
        # free space, ten thousand springs, stored weights, one radiation projection in each pass
        dict(name="free_1e4", kind="march", bc=FREE, M=10_000, layout="uniform", dt=1e-3, tol=1e-12, p=8, R=8, steps=54, lead=54),
        # one step at a time with the caller's forcing vector, densities and receivers read after each:
        # a march coupled to a program of the user's own
        dict(name="driven_step_2500", kind="step", bc=FREE, M=2_500, layout="uniform", dt=1e-3, tol=1e-12, p=6, R=5, lead=40),
        # the adjoint workload's medium marched forward: 1e5 springs, one implicit block, no pair lists
        dict(name="free_1e5", kind="march", bc=FREE, M=100_000, layout="uniform", dt=1e-3, tol=1e-12, p=8, R=8, steps=2, lead=42, local_weights=1),
        # the headline: a million springs, clustered, no pair lists
        dict(name="clustered_1e6", kind="march", bc=BOX, M=1_000_000, layout="clustered", clusters=16, dt=5e-4, tol=1e-10, p=4, R=4, steps=1, lead=12, local_weights=1),
        # the same medium at a third of its size and an odd count, FP32 spreading and interpolation
        dict(name="mixed_clustered_333333", kind="march", bc=BOX, M=333_333, layout="clustered", clusters=5, dt=5e-4, tol=1e-6, p=4, R=4, steps=2, lead=20, local_weights=1, precision=1),
        # dL/dbeta and dL/dg of a receiver misfit from stored densities, stored weights
        dict(name="gradient_6000", kind="gradient", bc=FREE, M=6_000, layout="uniform", dt=1e-3, tol=1e-12, p=8, R=8, steps=100),
        # the same from checkpoints through the plan without pair lists: the forward march again, then the reverse
        dict(name="gradient_ckpt_30000", kind="gradient", bc=FREE, M=30_000, layout="uniform", dt=1e-3, tol=1e-12, p=8, R=8, steps=10, interval=5, local_weights=1),
        # independent instances of very different sizes marched together, the form chosen per instance
        dict(name="batch_40", kind="batch", instances=40, lo=100, hi=30_000, dt=1e-3, tol=1e-12, p=8, steps=4, lead=42),
        # the history part's transforms alone at the headline's size, FP64
        dict(name="nufft_1e6", kind="nufft", M=1_000_000, instances=1, layout="clustered", clusters=16, K=6283, tol=1e-10, precision=0),
        # the same over many point sets in FP32 (the batched form)
        dict(name="nufft_many_mixed", kind="nufft", M=600_000, instances=64, layout="uniform", K=3141, tol=1e-6, precision=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["box", "free", "media", "step", "range", "clustered", "gradient", "gradient_ckpt", "batch", "nufft", "nufft_many"])
    if what == "box":
        return dict(kind="march", bc=BOX, M=_log(rng, 1, 900), layout="uniform", dt=rng.choice([0.01, 0.005]), tol=rng.choice([1e-8, 1e-10, 1e-12]),
                    p=rng.choice([4, 6, 8]), R=rng.randint(1, 9), steps=rng.randint(33, 96), lead=rng.randint(36, 64))
    if what == "free":
        return dict(kind="march", bc=FREE, M=_log(rng, 300, 9_000), layout="uniform", dt=rng.choice([1e-3, 1.5e-3]), tol=rng.choice([1e-10, 1e-12]),
                    p=rng.choice([4, 6, 8]), R=rng.randint(1, 16), steps=rng.randint(20, 54), lead=rng.randint(36, 60))
    if what == "media":
        return dict(kind="media", beta_max=rng.choice([3.0, 5.0, 10.0]), steps=rng.randint(30, 108), lead=rng.randint(150, 200))
    if what == "step":
        return dict(kind="step", bc=rng.choice([BOX, FREE]), M=_log(rng, 10, 6_000), layout="uniform", dt=1e-3, tol=rng.choice([1e-10, 1e-12]), p=rng.choice([4, 6]), R=rng.randint(1, 12), lead=rng.randint(20, 60))
    if what == "range":
        return dict(kind="march", bc=rng.choice([BOX, FREE]), M=_log(rng, 2_000, 100_000), layout="uniform", dt=1e-3, tol=rng.choice([1e-8, 1e-10, 1e-12]), p=rng.choice([4, 8]),
                    R=rng.randint(1, 8), steps=rng.randint(1, 3), lead=rng.randint(36, 44), local_weights=1)
    if what == "clustered":
        M = _log(rng, 20_000, 500_000)
        return dict(kind="march", bc=BOX, M=M, layout="clustered", clusters=max(1, round(M / 62_500)), dt=5e-4, tol=rng.choice([1e-8, 1e-10]), p=4,
                    R=rng.randint(1, 6), steps=rng.randint(1, 2), lead=rng.randint(12, 20), local_weights=1)
    if what == "gradient":
        return dict(kind="gradient", bc=rng.choice([BOX, FREE]), M=_log(rng, 100, 6_000), layout="uniform", dt=1e-3, tol=rng.choice([1e-10, 1e-12]), p=rng.choice([4, 6, 8]), R=rng.randint(1, 8), steps=rng.randint(40, 90))
    if what == "gradient_ckpt":
        return dict(kind="gradient", bc=FREE, M=_log(rng, 3_000, 30_000), layout="uniform", dt=1e-3, tol=1e-12, p=rng.choice([4, 8]), R=rng.randint(1, 8), steps=rng.randint(6, 10), interval=rng.randint(2, 6), local_weights=1)
    if what == "batch":
        return dict(kind="batch", instances=rng.randint(5, 40), lo=_log(rng, 10, 200), hi=_log(rng, 2_000, 20_000), dt=1e-3, tol=rng.choice([1e-10, 1e-12]), p=rng.choice([4, 8]), steps=rng.randint(2, 4), lead=rng.randint(36, 42))
    if what == "nufft":
        return dict(kind="nufft", M=_log(rng, 1_000, 1_000_000), instances=1, layout=rng.choice(["uniform", "clustered"]), clusters=16, K=_log(rng, 300, 6_283), tol=rng.choice([1e-8, 1e-10, 1e-12]), precision=0)
    return dict(kind="nufft", M=_log(rng, 20_000, 600_000), instances=rng.randint(2, 64), layout="uniform", K=_log(rng, 300, 3_141), tol=rng.choice([1e-5, 1e-6]), precision=1)


# --- inputs ------------------------------------------------------------------------------------
def _seed(seed):
    return (int(seed) * 1_000_003 + 7823) % (1 << 31)


def _workload(case, seed):
    """The springs, stiffnesses, pulses and receivers of a march."""
    if case["kind"] == "media":
        return workloads.disordered_media(case["beta_max"], seed=_seed(seed), Nt=1 << 40)
    kw = dict(M=case["M"], bc=case["bc"], dt=case["dt"], Nt=1 << 40, tol=case["tol"], p=case["p"], seed=_seed(seed), layout=case["layout"],
              beta_range=(0.1, 3.0), R=case["R"], margin=0.2)
    if case["layout"] == "clustered":
        kw.update(n_clusters=case["clusters"])
    # the pulses are drawn after the springs: `make` keeps springs away from those that it is given
    w = workloads.make("case", **kw, amp=(), center=(), width=())
    rng = np.random.Generator(np.random.PCG64(_seed(seed) + 1))
    return w.with_(amp=rng.uniform(0.3, 1.0, 3), center=rng.uniform(-2.0, 2.0, 3), width=rng.uniform(0.5, 1.0, 3))


def _batch_workloads(case, seed):
    rng = np.random.Generator(np.random.PCG64(_seed(seed)))
    # sizes evenly over their logarithm (the batch is as large for every seed), positions from the seed
    ms = np.exp(np.linspace(math.log(case["lo"]), math.log(case["hi"]), case["instances"])).astype(int)
    out = []
    for i, m in enumerate(ms):
        w = workloads.make(f"instance_{i}", M=int(m), bc=BOX, dt=case["dt"], Nt=1 << 40, tol=case["tol"], p=case["p"], seed=_seed(seed) + 11 * i + 1,
                           beta_range=(0.1, 3.0), amp=(), center=(), width=(), R=4)
        out.append(w.with_(amp=np.array([1.0]), center=rng.uniform(-2.0, 2.0, 1), width=rng.uniform(0.5, 1.0, 1)))
    return out


def _point_sets(case, seed):
    n, M = case["instances"], case["M"]
    if n == 1:
        sizes = [M]
    else:
        s = np.exp(np.linspace(math.log(1.0), math.log(300.0), n))
        sizes = np.maximum(1, (s * M / s.sum()).astype(int)).tolist()
    kw = dict(n_clusters=case["clusters"]) if case["layout"] == "clustered" else {}
    return [workloads.make("points", M=m, bc=BOX, dt=1e-3, Nt=1, seed=_seed(seed) + i, layout=case["layout"], amp=(), center=(), width=(), R=1, **kw).x for i, m in enumerate(sizes)]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(_seed(seed))


def _options(case):
    return {k: case[k] for k in ("local_weights", "precision") if k in case}


def _forcing(case, w, seed):
    """The caller's forcing vectors of the driven steps, one period of 20 steps."""
    g = _gen(seed)
    phase = 2 * math.pi * torch.rand(w.M, device="cuda", dtype=torch.float64, generator=g)
    beta = torch.from_numpy(w.beta).cuda()
    return [beta * torch.cos(2 * math.pi * i / 20 + phase) for i in range(20)]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("march", "media"):
        w = _workload(case, seed)
        plan = wave1d.Plan.from_workload(w, **_options(case))
        _march(plan, case["lead"])
        return dict(case=case, plan=plan)
    if kind == "step":
        w = _workload(case, seed)
        plan = wave1d.Plan.from_workload(w, **_options(case))
        state = dict(case=case, plan=plan, g=_forcing(case, w, seed), n=0)
        for _ in range(case["lead"]):
            _driven(state)
        return state
    if kind == "gradient":
        w = _workload(case, seed)
        plan = wave1d.Plan.from_workload(w, **_options(case))
        ubar = torch.randn(case["steps"], case["R"], device="cuda", dtype=torch.float64, generator=_gen(seed))
        if "interval" in case:
            _, ckpt = plan.solve_checkpointed(case["steps"], case["interval"])
            return dict(case=case, plan=plan, ubar=ubar, ckpt=ckpt)
        sigma, _ = plan.solve_device(case["steps"])
        return dict(case=case, plan=plan, ubar=ubar, sigma=sigma)
    if kind == "batch":
        batch = wave1d.Batch(_batch_workloads(case, seed), local_weights=2)
        batch.solve(case["lead"], with_sigma=False)
        return dict(case=case, batch=batch)
    sets = _point_sets(case, seed)
    plan = wave1d.Nufft(sets if case["instances"] > 1 else sets[0], case["K"], case["tol"], case["precision"])
    c, alpha = _coefficients(case, plan.M, seed)
    return dict(case=case, plan=plan, c=c, alpha=alpha, S=torch.empty_like(alpha), u=torch.empty_like(c))


def _march(plan, n):
    """n steps of a march whose densities nobody reads."""
    u = torch.empty((n, max(plan.R, 1)), dtype=torch.float64, device="cuda")
    st = wave1d.wave1d_solve(plan.h, n, u, None, 1)
    if st != wave1d.WAVE1D_OK:
        raise wave1d.Wave1DError(st, "wave1d_solve")


def _coefficients(case, M, seed):
    g = _gen(seed)
    c = torch.randn(M, device="cuda", dtype=torch.float64, generator=g)
    a = torch.randn(case["instances"], case["K"] + 1, 2, device="cuda", dtype=torch.float64, generator=g)
    a[:, 0, 1] = 0.0
    return c, a


def _driven(state):
    plan, g = state["plan"], state["g"]
    wave1d._check(wave1d.wave1d_step(plan.h, g[state["n"] % len(g)], 1), "wave1d_step")
    state["n"] += 1


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("march", "media"):
        return state["plan"].solve_device(case["steps"])
    if kind == "step":
        plan = state["plan"]
        _driven(state)
        sigma = torch.empty(plan.M, dtype=torch.float64, device="cuda")
        u = torch.empty(plan.R, dtype=torch.float64, device="cuda")
        wave1d._check(wave1d.wave1d_get_sigma(plan.h, sigma, 1), "wave1d_get_sigma")
        wave1d._check(wave1d.wave1d_read_receivers(plan.h, u, 1), "wave1d_read_receivers")
        return sigma, u
    if kind == "gradient":
        if "interval" in case:
            return state["plan"].adjoint_checkpointed(state["ckpt"], case["steps"], case["interval"], state["ubar"], forcing_gradient=True)
        return state["plan"].adjoint(state["sigma"], state["ubar"], forcing_gradient=True)
    if kind == "batch":
        return state["batch"].solve(case["steps"])
    plan = state["plan"]
    plan.type1(state["c"], state["S"])
    plan.type2(state["alpha"], state["u"])
    return state["S"], state["u"]


# --- work ---------------------------------------------------------------------------------------
def _march_work(M, dt, tol, p, R, box_fraction, near):
    """Bytes and multiply-adds of one step: the density history within the window read once and the new densities
    written, and the terms of the local sum (pairs within delta, on average half of the window's steps each), the
    FIR sums of the modes and the two transforms by FFT."""
    W = math.ceil(4.0 * math.log(1.0 / tol) / math.pi)
    K = int(math.pi / dt)
    pairs = M * min(1.0, near * 2 * W * dt) * M
    terms = pairs * 0.5 * (W + p) + 2.0 * W * 2 * (K + 1) + 20.0 * M
    return 8.0 * M * (W + p // 2 + 4) + 16.0 * 3 * W * (K + 1) + 8.0 * R, 2.0 * terms + 10.0 * K * math.log2(4 * K)


def work(case):
    kind = case["kind"]
    if kind == "media":
        b, f = _march_work(150, 3.703e-3, 1e-12, 8, 100, 1.0, 1 / 4.0)
        return dict(bytes=case["steps"] * b, flops=case["steps"] * f)
    if kind in ("march", "step", "gradient"):
        # a clustered layout: four fifths of the springs in clusters of width 0.05, about three widths long each
        near = 1 / (2 * math.pi) if case["layout"] == "uniform" else 0.64 / (case["clusters"] * 0.05 * 2 * math.sqrt(math.pi))
        b, f = _march_work(case["M"], case["dt"], case["tol"], case["p"], case["R"], 1.0, near)
        n = case.get("steps", 1) * (2 if "interval" in case else 1)
        return dict(bytes=n * b, flops=n * f)
    if kind == "batch":
        ms = np.exp(np.linspace(math.log(case["lo"]), math.log(case["hi"]), case["instances"])).astype(int)
        bf = [_march_work(int(m), case["dt"], case["tol"], case["p"], 4, 1.0, 1 / (2 * math.pi)) for m in ms]
        return dict(bytes=case["steps"] * sum(b for b, _ in bf), flops=case["steps"] * sum(f for _, f in bf))
    M, K, n = case["M"], case["K"], case["instances"]
    taps = math.ceil(math.log10(1 / case["tol"])) + 1
    return dict(bytes=4.0 * 8 * M + 2.0 * 16 * n * (K + 1), flops=2 * (2.0 * taps * M + n * 10.0 * K * math.log2(4 * K)))


# --- the same in 64 bits, plainly ----------------------------------------------------------------
# The discrete scheme of the windowed Fourier projection method restated in torch: direct Fourier sums, the local
# weights from their quadrature, dense solves.  Only for cases that take seconds this way.
class _Scheme:
    def __init__(self, x, beta, box, dt, tol, p, pulses, xr):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        T = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=self.dev)  # noqa: E731
        self.x, self.beta, self.xr, self.box, self.dt, self.p = T(x), T(beta), T(xr), box, dt, p
        self.pulses = pulses
        b = math.log(1.0 / tol)
        self.K, self.W = int(math.floor(math.pi / dt)), int(math.ceil(4.0 * b / math.pi))
        self.m_max = self.W + (p + 1) // 2
        self.delta, self.b, self.period = self.W * dt, b, int(math.ceil(1.5 * self.W))
        K, W = self.K, self.W
        k = torch.arange(K + 1, device=self.dev, dtype=torch.float64)
        self.weights = torch.where(k == 0, 1.0, 2.0)
        self.E = torch.exp(1j * self.x[:, None] * k)
        self.Er = torch.exp(-1j * self.xr[:, None] * k)
        # p_k, q_k by Gauss-Legendre
        gx, gw = np.polynomial.legendre.leggauss(32)
        mu, wt = T(0.5 * dt * (1 + gx)), T(0.5 * dt * gw)
        kk = k[None, :, None]
        sk = lambda t: torch.where(kk == 0, t, torch.sin(kk * t) / torch.where(kk == 0, 1.0, kk))  # noqa: E731
        pk, qk = [], []
        for m in range(W):
            tau = (m * dt + mu)[None, None, :]
            psi = 2 * torch.cos(kk * tau) * self.dphi(tau, self.delta) + sk(tau) * self.ddphi(tau, self.delta)
            pk.append((wt * sk(dt - mu) * psi).sum(-1)[0])
            qk.append((wt * torch.cos(kk * (dt - mu)) * psi).sum(-1)[0])
        self.pk, self.qk = dt * torch.stack(pk), dt * torch.stack(qk)
        self.rot = (torch.cos(k * dt), torch.where(k == 0, dt, torch.sin(k * dt) / torch.where(k == 0, 1.0, k)), k * torch.sin(k * dt))
        self.cheb = {w: self.window_series(w) for w in (self.delta, W * math.pi / K)}
        # local weights of springs (m >= 1 sparse, m = 0 dense) and of receivers
        M = len(self.x)
        C, Q0 = self.stack(self.x, 1)
        self.C, self.Q0 = C, Q0
        self.Ct = C.t().to_sparse_csr()
        self.lu = torch.linalg.lu_factor(torch.eye(M, device=self.dev, dtype=torch.float64) + 0.5 * self.beta[:, None] * Q0)
        self.Cr = self.stack(self.xr, 0)[0] if len(self.xr) else None
        self.Crt = self.Cr.t().to_sparse_csr() if len(self.xr) else None

    # the blending window of a given width
    def dphi(self, t, width):
        u = 2 * t / width - 1
        z = self.b * torch.sqrt(torch.clamp(1 - u * u, min=0))
        return torch.where((t >= 0) & (t <= width), self.b / (width * math.sinh(self.b)) * torch.special.i0(z), 0.0)

    def ddphi(self, t, width):
        u = 2 * t / width - 1
        z = self.b * torch.sqrt(torch.clamp(1 - u * u, min=0))
        r = torch.where(z > 1e-8, torch.special.i1(z) / torch.clamp(z, min=1e-8), 0.5)
        return torch.where((t >= 0) & (t <= width), -(2 * self.b ** 3 * u / (width * width * math.sinh(self.b))) * r, 0.0)

    def window_series(self, width):
        gx, gw = np.polynomial.legendre.leggauss(96)

        def quad(z):
            t = 0.25 * width * (np.asarray(z) + 1.0)
            s = torch.as_tensor(0.5 * t[:, None] * (1 + gx))
            return 0.5 * t * (gw * self.dphi(s, width).numpy()).sum(-1)
        return np.polynomial.chebyshev.chebinterpolate(quad, 48)

    def phi(self, t, width):
        tc = torch.clamp(t, 0.0, width)
        low = tc <= 0.5 * width
        z = 4 * torch.where(low, tc, width - tc) / width - 1
        b1 = b2 = torch.zeros_like(z)
        for c in self.cheb[width][:0:-1]:
            b1, b2 = 2 * z * b1 - b2 + float(c), b1
        v = z * b1 - b2 + float(self.cheb[width][0])
        return torch.where(t <= 0, 0.0, torch.where(t >= width, 1.0, torch.where(low, v, 1 - v)))

    def stack(self, targets, first):
        """Sparse rows of Q_m over [sigma^{n+1-first}, sigma^{n-first}, ...], and the dense Q_0 if first = 1."""
        M, ti, si, di = len(self.x), [], [], []
        for a in range(0, len(targets), 512):
            d = (targets[a:a + 512, None] - self.x).abs()
            if self.box:
                d = torch.remainder(d, 2 * math.pi)
                d = torch.minimum(d, 2 * math.pi - d)
            t, s = torch.nonzero(d < self.delta, as_tuple=True)
            ti.append(t + a), si.append(s), di.append(d[t, s])
        t, s, d = torch.cat(ti), torch.cat(si), torch.cat(di)
        Q = torch.cat([self.local_weights(d[a:a + 200_000]) for a in range(0, len(d), 200_000)]) if len(d) else torch.zeros(0, self.m_max + 1, device=self.dev, dtype=torch.float64)
        Q0 = None
        if first:
            Q0 = torch.zeros(len(targets), M, device=self.dev, dtype=torch.float64)
            Q0.index_put_((t, s), Q[:, 0], accumulate=True)
        e, m = torch.nonzero(Q[:, first:], as_tuple=True)
        C = torch.sparse_coo_tensor(torch.stack([t[e], m * M + s[e]]), Q[e, m + first], (len(targets), (self.m_max + 1 - first) * M)).coalesce()
        return C.to_sparse_csr(), Q0

    def local_weights(self, d):
        gx, gw = (torch.as_tensor(v, device=self.dev) for v in np.polynomial.legendre.leggauss(self.W))
        half = 0.5 * (self.delta - d)[:, None]
        s = d[:, None] + half * (1 + gx)
        wphi = half * gw * (1 - self.phi(s, self.delta))
        y = s / self.dt
        lo = torch.floor(y).long() - self.p // 2 + 1
        lo = torch.maximum(lo, torch.where(d < self.dt, 0, 1)[:, None])
        lo = torch.clamp(lo, max=self.m_max - self.p + 1)
        Q = torch.zeros(len(d), self.m_max + 1, device=self.dev, dtype=torch.float64)
        for r in range(self.p):
            L = torch.ones_like(y)
            for q in range(self.p):
                if q != r:
                    L = L * (y - (lo + q)) / (r - q)
            Q.scatter_add_(1, lo + r, wphi * L)
        return Q

    def project(self, a, ap):
        """The radiation projection on a grid of 2 K points."""
        K, W, n, ds = self.K, self.W, 2 * self.K, self.W * math.pi / self.K

        def grid(v):
            z = torch.zeros((), device=self.dev, dtype=v.dtype)
            return torch.fft.fft(torch.cat([v[:K], z[None], torch.conj(v[1:K]).flip(0)])).real
        u, v = grid(a), grid(ap)
        i = torch.arange(n, device=self.dev)
        xg = torch.where(i < K, i, i - n) * (math.pi / K)
        for idx, sign in ((i[K - 2 * W:K], -1.0), (i[K:K + 2 * W], 1.0)):
            arg = math.pi - ds + sign * xg[idx]
            ph, dph = self.phi(arg, ds), self.dphi(arg, ds)
            un, vn = u.clone(), v.clone()
            un[idx], vn[idx] = ph * u[idx], dph * u[idx] + ph * v[idx]
            u, v = un, vn
        keep = torch.arange(K + 1, device=self.dev) < K
        return tuple(torch.where(keep, torch.fft.ifft(w.to(a.dtype))[:K + 1], 0) for w in (u, v))

    def incident(self, t):
        f = torch.zeros_like(self.x)
        for amp, c, w in self.pulses:
            for m in (range(-4, 5) if self.box else (0,)):
                f = f + amp * torch.exp(-0.5 * ((self.x - t + 2 * math.pi * m - c) / w) ** 2)
        return f

    def march(self, steps, forcing=None, beta=None):
        """All densities and receiver fields of `steps` steps from rest, differentiable in `beta` and `forcing`."""
        beta = self.beta if beta is None else beta
        M, zero = len(self.x), torch.zeros_like(self.x)
        sig, S = [zero] * (self.m_max + 1), []
        a = ap = torch.zeros(self.K + 1, device=self.dev, dtype=torch.complex128)
        sigmas, us = [], []
        for n in range(steps):
            S = [(sig[0].to(a.dtype) @ self.E) / (2 * math.pi)] + S[:self.W - 1]
            St = torch.stack(S)
            h, g = (self.pk[:len(S)] * St).sum(0), (self.qk[:len(S)] * St).sum(0)
            c, so, ks = self.rot
            a, ap = a * c + ap * so + h, -a * ks + ap * c + g
            if not self.box and (n + 1) % self.period == 0:
                a, ap = self.project(a, ap)
            uH = (torch.conj(self.E) @ (self.weights * a)).real
            local = _Spmv.apply(self.C, self.Ct, torch.cat(sig[:self.m_max]))
            gn = beta * self.incident((n + 1) * self.dt) if forcing is None else forcing[n]
            new = _Solve.apply(self.lu, self.Q0, -gn - 0.5 * beta * local - beta * uH, beta)
            sig = [new] + sig[:-1]
            sigmas.append(new)
            if self.Cr is not None:
                us.append(0.5 * _Spmv.apply(self.Cr, self.Crt, torch.cat(sig)) + (self.Er @ (self.weights * a)).real)
        return torch.stack(sigmas), torch.stack(us)


class _Spmv(torch.autograd.Function):
    @staticmethod
    def forward(ctx, A, At, v):
        ctx.At = At
        return A @ v

    @staticmethod
    def backward(ctx, g):
        return None, None, ctx.At @ g


class _Solve(torch.autograd.Function):
    """sigma of (I + diag(beta / 2) Q_0) sigma = rhs."""
    @staticmethod
    def forward(ctx, lu, Q0, rhs, beta):
        s = torch.linalg.lu_solve(*lu, rhs[:, None])[:, 0]
        ctx.lu, ctx.Q0, ctx.s = lu, Q0, s
        return s

    @staticmethod
    def backward(ctx, g):
        r = torch.linalg.lu_solve(*ctx.lu, g[:, None], adjoint=True)[:, 0]
        return None, None, r, -0.5 * r * (ctx.Q0 @ ctx.s)


def _scheme(case, seed):
    w = _workload(case, seed)
    return w, _Scheme(w.x, w.beta, w.bc == BOX, w.dt, w.tol, w.p, list(zip(w.amp, w.center, w.width)), w.xr)


def exact(case, seed):
    kind = case["kind"]
    if kind == "nufft":
        if case["instances"] > 1 and case["M"] * case["K"] > 2.5e9:
            return None
        return _exact_nufft(case, seed)
    # the plan without pair lists is for layouts whose pairs a plain program cannot hold; a batch is many plans
    if kind == "batch" or case.get("local_weights"):
        return None
    w, s = _scheme(case, seed)
    if kind in ("march", "media"):
        with torch.no_grad():
            sigma, u = s.march(case["lead"] + case["steps"])
        return sigma[case["lead"]:], u[case["lead"]:]
    if kind == "step":
        g = _forcing(case, w, seed)
        with torch.no_grad():
            sigma, u = s.march(case["lead"] + 1, [g[n % len(g)] for n in range(case["lead"] + 1)])
        return sigma[-1], u[-1]
    ubar = torch.randn(case["steps"], case["R"], device="cuda", dtype=torch.float64, generator=_gen(seed))
    beta = s.beta.clone().requires_grad_(True)
    # dL/dg at the incident wave's own forcing, dL/dbeta through the whole march
    slack = torch.zeros(case["steps"], w.M, device=s.dev, dtype=torch.float64, requires_grad=True)
    forcing = [beta * s.incident((n + 1) * s.dt) + slack[n] for n in range(case["steps"])]
    _, u = s.march(case["steps"], forcing, beta)
    return torch.autograd.grad((u * ubar).sum(), (beta, slack))


def _exact_nufft(case, seed):
    """Direct sums over the points, each set's points in the plan's order (sorted by first fine-grid cell, then position)."""
    sets, K, tol = _point_sets(case, seed), case["K"], case["tol"]
    taps = max(4, math.ceil(math.log10(1 / tol)) + 1)
    nf = 1 << max(6, math.ceil(math.log2(2 * (2 * K + 1))))
    c, alpha = _coefficients(case, sum(len(v) for v in sets), seed)
    k = torch.arange(K + 1, device="cuda", dtype=torch.float64)
    S, u, at = [], [], 0
    for i, x in enumerate(sets):
        first = np.ceil((x + math.pi) / (2 * math.pi / nf) - 0.5 * taps).astype(int) % nf
        x = torch.from_numpy(x[np.lexsort((x, first))]).cuda()
        ci, a = c[at:at + len(x)], torch.view_as_complex(alpha[i])
        wa = torch.where(k == 0, 1.0, 2.0) * a
        Sk, step = torch.zeros(K + 1, device="cuda", dtype=torch.complex128), max(1, 40_000_000 // (K + 1))
        for j in range(0, len(x), step):
            ph = x[j:j + step, None] * k
            cs, sn = torch.cos(ph), torch.sin(ph)
            Sk += torch.complex(ci[j:j + step] @ cs, ci[j:j + step] @ sn)
            u.append(cs @ wa.real + sn @ wa.imag)
        S.append(torch.view_as_real(Sk / (2 * math.pi)))
        at += len(x)
    return torch.stack(S), torch.cat(u)
