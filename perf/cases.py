"""The work that users of this library run on one GPU, as timed cases.

Every case is one short pulse run through the public classes: the bare-mode
engines (``LowRankBatch``), the sparse-operator engine and the full master
equation on the paper's normal-mode model (``SparseBatch``, ``FullME``), and
the gradient of the assignment error (``assignment_error``). A full pulse is
80,000 RK4 steps; a case runs the first few dozen to few hundred of a pulse
scaled to that length, which cost the same per step.

The engines hand out doubles. Where the state is FP32 a program keeps them as
the float32 numbers that they are, and so does ``run``.

``exact`` integrates the same equation (Eq. S5 of arXiv 2508.18114, or Eq. 2 for
the full master equation) in complex128 with plain torch operations: ladder
operators by slicing, a Cholesky solve of the Gram matrix, classical RK4.
"""
import math
import random

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2508_18114_gb300 import LowRankBatch
from paper_2508_18114_gb300.autograd import assignment_error
from paper_2508_18114_gb300.sparse import FullME, SparseBatch, paper_model

TWO_PI = 2.0 * math.pi
EPS = 1e-5          # weight of each padding column of the initial state
ETA = 0.6           # measurement efficiency
KAPPA, GAMMA = TWO_PI * 0.05, 1.0 / 50000.0
OMEGA_MAX = TWO_PI * 0.4


class Model:
    """Bare-mode transmon x resonator (x filter) model of the given cutoffs."""

    def __init__(self, dims):
        self.dims = tuple(dims)
        self.wq, self.alpha, self.wr = TWO_PI * 6.0, -TWO_PI * 0.3, TWO_PI * 7.5
        self.g, self.kappa, self.gamma = TWO_PI * 0.15, KAPPA, GAMMA
        self.wf, self.J = self.wr + TWO_PI * 0.01, TWO_PI * 0.1


def paper_params():
    """Parameters of the paper's Sec. S2.B (rad/ns, 1/ns)."""
    ec = TWO_PI * 0.315
    return dict(Ec=ec, Ej=51.0 * ec, wr=TWO_PI * 7.2, wf=TWO_PI * 7.21, g=TWO_PI * 0.15, J=TWO_PI * 0.03,
                kappa=TWO_PI * 0.03, gamma=TWO_PI * 8e-6, wd=TWO_PI * 7.18)


# ------------------------------------------------------------------- cases --
def listed():
    return [
        # one candidate on the small two-mode model: interactive use, pure latency
        dict(name="single_small_fp64", kind="batch", dims="4x10", M=4, cands=1, steps=400, dt=1e-3,
             precision="fp64", frame="lab", pop_every=40, uneven=0),
        # one candidate of the N = 2000 model in FP64: a reference trajectory,
        # resumed from a checkpoint and checkpointed again
        dict(name="single_fp64_resume", kind="resume", dims="10x20x10", M=20, cands=1, steps=40, dt=5e-4,
             precision="fp64", frame="lab", pop_every=10, uneven=0),
        # the same model in production precision: one pulse evaluated alone
        dict(name="single_fp32", kind="batch", dims="10x20x10", M=20, cands=1, steps=240, dt=5e-4,
             precision="fp32_g64", frame="lab", pop_every=20, uneven=0),
        # a population of 256 pulse candidates per launch: the outer loop of a pulse search
        dict(name="population_fp32", kind="batch", dims="10x20x10", M=20, cands=256, steps=64, dt=5e-4,
             precision="fp32_g64", frame="lab", pop_every=16, uneven=0),
        # a population of designs with uneven cutoffs and ranks
        dict(name="uneven_fp32", kind="batch", dims="12x30x12", M=30, cands=128, steps=24, dt=5e-4,
             precision="fp32_g64", frame="lab", pop_every=8, uneven=11),
        # the large model at the highest rank
        dict(name="large_rank_fp32", kind="batch", dims="10x40x20", M=32, cands=64, steps=16, dt=5e-4,
             precision="fp32_g64", frame="lab", pop_every=8, uneven=0),
        # a medium population in the rotating frame, the larger step of the RWA
        dict(name="population_rwa", kind="batch", dims="10x20x10", M=20, cands=76, steps=100, dt=2.5e-3,
             precision="fp32_g64", frame="rwa", pop_every=20, uneven=0),
        # gradient of the assignment error with respect to every pulse parameter, in
        # the precision that resolves it (|beta_e - beta_g| is small early in a pulse)
        dict(name="gradient_fp64", kind="gradient", dims="10x20x10", M=20, cands=6, steps=16, dt=5e-4,
             precision="fp64", frame="lab", pop_every=8, uneven=0),
        # the paper's own model: a population of pulses, production precision
        dict(name="paper_population", kind="sparse", dims="100x4x5", M=20, cands=256, steps=40, dt=5e-4,
             precision="fp32_g64", frame="rot", pop_every=10, uneven=0),
        # the paper's Fig. 2: one pulse, |g> and |e>
        dict(name="paper_single", kind="sparse", dims="100x4x5", M=20, cands=1, steps=240, dt=5e-4,
             precision="fp32_g64", frame="rot", pop_every=20, uneven=0),
        # the same model in FP64 for a check of a few pulses
        dict(name="paper_fp64", kind="sparse", dims="100x4x5", M=20, cands=16, steps=16, dt=5e-4,
             precision="fp64", frame="rot", pop_every=8, uneven=0),
        # the full master equation the low-rank runs are compared with
        dict(name="full_master_equation", kind="full", dims="100x4x5", M=1, cands=1, steps=6, dt=5e-4,
             precision="fp64", frame="rot", pop_every=2, uneven=0),
    ]


def _step_cost(kind, N, M, traj, precision):
    """A rough cost of one RK4 step in seconds, to keep drawn cases short."""
    if kind == "full":
        return 6e-3 * (N / 2000.0) ** 2 + 4e-4
    work = N * M * (M + 11.0) / 1.24e6
    if kind == "gradient":
        return max(traj * work / 7e2, 1e-2 * max(0.5, (M / 20.0) ** 2))
    if precision == "fp64":
        return max(traj * work / 4.5e3, 1.7e-3 * max(0.5, (M / 20.0) ** 2))
    return max(traj * work / 8e4, 3.5e-4 * max(1.0, M / 20.0))


def draw(rng):
    """Another case of the same ranges."""
    kind = rng.choice(["batch", "batch", "batch", "batch", "sparse", "sparse", "resume", "gradient", "full"])
    frame, precision, uneven = "lab", "fp32_g64", 0
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    cands = log(1, 256)
    if kind in ("sparse", "full"):
        dims = (rng.randint(20, 100), rng.randint(2, 6), rng.randint(3, 6))
        frame = rng.choice(["rot", "rot", "rwa"])
        M = log(4, 32)
        if kind == "full":
            cands, M, precision = 1, 1, "fp64"
        elif rng.random() < 0.3:
            precision, cands = "fp64", log(1, 16)
    else:
        two = rng.random() < 0.2
        dims = (rng.randint(4, 12), rng.randint(10, 40)) if two else (rng.randint(4, 12), rng.randint(10, 40),
                                                                       rng.randint(5, 20))
        M = log(4, 32)
        if kind == "batch":
            if rng.random() < 0.25:
                precision, cands = "fp64", log(1, 32)
            elif rng.random() < 0.3:
                frame = "rwa"
            if not two and cands > 1 and rng.random() < 0.3:
                uneven, dims, M = rng.randint(1, 10 ** 6), (12, 30, 12), 30
        elif kind == "resume":
            precision, cands = rng.choice(["fp64", "fp32_g64"]), 1
        else:
            precision, cands = "fp64", log(1, 8)
    N = int(np.prod(dims))
    M = min(M, N)
    dt = 2.5e-3 if frame == "rwa" else 5e-4
    cost = _step_cost(kind, N, M, 2 * cands, precision)
    steps = max(3, min(200, int(0.18 / cost)))
    while steps == 3 and cost * 3 > 0.3 and cands > 1:
        cands = max(1, cands // 2)
        cost = _step_cost(kind, N, M, 2 * cands, precision)
    return dict(kind=kind, dims="x".join(str(d) for d in dims), M=M, cands=cands, steps=steps, dt=dt,
                precision=precision, frame=frame, pop_every=max(1, steps // 4), uneven=uneven)


def _sizes(case):
    """(dims, rank) of every candidate."""
    dims = tuple(int(x) for x in case["dims"].split("x"))
    if not case["uneven"]:
        return [(dims, case["M"])] * case["cands"]
    r = random.Random(case["uneven"])
    return [((r.randint(6, 12), r.randint(15, 30), r.randint(8, 12)), r.randint(10, 30)) for _ in range(case["cands"])]


def _pulses(case, seed):
    """(kind, parameters) per candidate: a pulse that fills the run's window,
    with the edges scaled to its length."""
    r = random.Random(1000003 * seed + 17)
    tau = case["steps"] * case["dt"]
    wr = paper_params()["wr"] if case["kind"] in ("sparse", "full") else TWO_PI * 7.5
    out = []
    for _ in range(case["cands"]):
        a1 = OMEGA_MAX * r.uniform(0.1, 1.0)
        wd = r.uniform(wr - TWO_PI * 0.03, wr + TWO_PI * 0.03)
        phi = r.uniform(0.0, TWO_PI)
        if case["kind"] in ("sparse", "full"):
            out.append((0, (a1, paper_params()["wd"], tau * r.uniform(0.1, 0.3), 0.0)))
        elif case["M"] <= 8:
            out.append((0, (a1, wd, tau * r.uniform(0.1, 0.3), phi)))
        else:
            out.append((1, (a1, a1 * r.uniform(0.1, 1.0), tau * r.uniform(0.3, 0.7), tau * r.uniform(0.1, 0.3),
                            tau * r.uniform(0.1, 0.3), tau * r.uniform(0.1, 0.3), wd, phi)))
    return out


def _start_state(case, seed):
    """A checkpoint of one trajectory: a dominant state and decaying columns."""
    (dims, M), = set(_sizes(case))
    N = int(np.prod(dims))
    g = np.random.default_rng(seed)
    z = g.standard_normal((2, N, M)) + 1j * g.standard_normal((2, N, M))
    q = np.stack([np.linalg.qr(m)[0] for m in z])
    p = 10.0 ** -np.linspace(0.0, 5.0, M)
    return q * np.sqrt(p / p.sum())


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, s.seed, s.pulses, s.tau = case, int(seed), _pulses(case, seed), case["steps"] * case["dt"]
    dims = tuple(int(x) for x in case["dims"].split("x"))
    if case["kind"] in ("sparse", "full"):
        s.model = paper_model(*dims, frame=case["frame"], **paper_params())
        if case["kind"] == "full":
            s.me = FullME(s.model, s.pulses[0], s.tau, case["steps"], pop_every=case["pop_every"])
            return s
        s.pulses2 = [p for p in s.pulses for _ in range(2)]
        s.psi = [0, 1] * case["cands"]
        s.batch = SparseBatch(s.model, case["M"], s.pulses2, s.tau, case["steps"], pop_every=case["pop_every"],
                              precision=case["precision"])
        return s
    sizes = _sizes(case)
    s.batch = LowRankBatch([Model(d) for d, _ in sizes], [m for _, m in sizes], precision=case["precision"],
                           max_steps=case["steps"], pop_every=case["pop_every"], eta=ETA, frame=case["frame"])
    if case["kind"] == "resume":
        s.batch.set_pulse(s.pulses, s.tau)
        s.z0 = _start_state(case, seed)
    if case["kind"] == "gradient":
        th = np.zeros((case["cands"], 8))
        for c, (_, p) in enumerate(s.pulses):
            th[c, :len(p)] = p
        s.theta = torch.from_numpy(th)
        s.weights = torch.from_numpy(np.random.default_rng(seed).uniform(0.5, 1.5, case["cands"]))
    return s


def _kept(case, out):
    """The observables in the precision of the run (float32 for an FP32 state)."""
    if case["precision"] == "fp64":
        return out
    return {k: np.asarray(v).astype(np.complex64 if np.iscomplexobj(v) else np.float32) for k, v in out.items()}


def run(s):
    case = s.case
    dt, n = case["dt"], case["steps"]
    if case["kind"] == "full":
        s.me.set_initial(1)
        s.me.integrate(dt, n)
        out = dict(s.me.observables())
        out["rho"] = s.me.get_state()
        return out
    if case["kind"] == "sparse":
        s.batch.set_initial(s.psi, s.seed, EPS)
        s.batch.integrate(dt, n)
        out = dict(s.batch.observables())
        p = paper_params()
        out.update(s.batch.loss(p["kappa"], p["gamma"], ETA))
        if case["cands"] == 1:        # a single pulse keeps its final state
            out["Z"] = s.batch.get_state()
        return _kept(case, out)
    if case["kind"] == "gradient":
        theta = s.theta.clone().requires_grad_(True)
        eps_a = assignment_error(theta, s.batch, [k for k, _ in s.pulses], s.tau, dt, n, s.seed, EPS, ckpt_every=10)
        (eps_a * s.weights).sum().backward()
        return _kept(case, {"eps_a": eps_a.detach().numpy(), "gradient": theta.grad.numpy()})
    if case["kind"] == "resume":
        for j in range(2):
            s.batch.set_state(j, s.z0[j], 0)
    else:
        s.batch.set_pulse(s.pulses, s.tau)
        s.batch.set_initial(s.seed, EPS)
    s.batch.integrate(dt, n)
    o = s.batch.observables()
    out = {k: o[k] for k in ("beta", "pops", "nphot", "trace", "eps_a")}
    out["ionization"], out["loss"] = s.batch.loss()
    if case["cands"] == 1:            # a single pulse keeps its final state
        out["Z"] = np.stack([s.batch.get_state(j) for j in range(2)])
    return _kept(case, out)


# -------------------------------------------------------------------- work --
def work(case):
    es = 16 if case["precision"] == "fp64" else 8
    byts, flops = 0, 0.0
    for dims, M in _sizes(case):
        N = int(np.prod(dims))
        stages = 4.0 * case["steps"]
        if case["kind"] == "full":
            # rho -> A rho, L_k rho and their adjoint products: about 24 entries
            # per row of the operators, one complex multiply-add each
            flops += stages * 24 * 8.0 * N * N
            byts += 16 * N * N
            continue
        nnz = 24 if case["kind"] == "sparse" else (11 if len(dims) == 3 else 7)
        per = 4.0 * N * M * M + 16.0 * N * M * M * 2 + (8.0 if case["kind"] == "sparse" else 4.0) * nnz * N * M + 12.0 * N * M
        # the reverse pass of a gradient is twice the forward work, after one
        # recomputation of the checkpointed steps
        flops += 2 * stages * per * (4.0 if case["kind"] == "gradient" else 1.0)
        # the records; a single pulse also returns its state, and reads it when resumed
        levels = dims[-1] if case["kind"] == "sparse" else dims[0]
        byts += 2 * ((case["steps"] + 1) * es + (case["steps"] // case["pop_every"] + 1) * (levels + 2) * es // 2)
        if case["cands"] == 1:
            byts += 2 * N * M * es * (2 if case["kind"] == "resume" else 1)
    return {"bytes": int(byts), "flops": float(flops)}


# ----------------------------------------------------------------- exact --
_MASK = (1 << 64) - 1


def _signed(x):
    x &= _MASK
    return x - (1 << 64) if x >> 63 else x


def _mix64(z):
    """SplitMix64's finalizer (Steele, Lea, Flood 2014) on int64 tensors."""
    shr = lambda v, k: (v >> k) & ((1 << (64 - k)) - 1)  # noqa: E731
    z = (z ^ shr(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * _signed(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _stream(seed, k):
    return _mix64(seed + (k + 1) * _signed(0x9E3779B97F4A7C15))


def _initial(dims, M, ts, levels, stride):
    """Z(0) [T, N, M]: psi with weight 1 - (M - 1) eps, and sqrt(eps) times the
    orthonormalised Gaussian columns; stride: rows per level of psi."""
    N, T = int(np.prod(dims)), len(levels)
    z = torch.zeros(T, N, M, dtype=torch.complex128, device="cuda")
    z[torch.arange(T), torch.tensor(levels) * stride, 0] = 1.0
    if M > 1:
        p = torch.arange((M - 1) * N, device="cuda", dtype=torch.int64)
        u = [(((_stream(ts[:, None], 2 * p + i) >> 11) & ((1 << 53) - 1)).double() + 1.0) * 2.0 ** -53 for i in (0, 1)]
        xi = torch.sqrt(-2.0 * torch.log(u[0])) * torch.exp(2j * math.pi * u[1])
        z[:, :, 1:] = xi.reshape(T, M - 1, N).transpose(1, 2)
        for _ in range(3):          # Gram-Schmidt by Cholesky QR, repeated to full precision
            chol = torch.linalg.cholesky(z.mH @ z)
            z = torch.linalg.solve_triangular(chol, z.mH, upper=False).mH.contiguous()
    w = torch.full((M,), math.sqrt(EPS), dtype=torch.float64, device="cuda")
    w[0] = math.sqrt(1.0 - (M - 1) * EPS)
    return z * w


def _shift(z, ax, up, mask):
    """a z (up False) or a^dag z (up True) of the mode on axis ax, truncated."""
    d = z.shape[ax]
    out = torch.zeros_like(z)
    w = torch.sqrt(torch.arange(1, d, dtype=torch.float64, device=z.device)).reshape([-1 if i == ax else 1 for i in range(z.dim())])
    if up:
        out.narrow(ax, 1, d - 1).copy_(w * z.narrow(ax, 0, d - 1))
    else:
        out.narrow(ax, 0, d - 1).copy_(w * z.narrow(ax, 1, d - 1))
    return out if mask is None else out * mask


def _logistic(t, t0, s):
    return torch.sigmoid((t - t0) / s)


def _envelope(pulse, tau, t):
    """Omega(t) of Sec. S2.C; pulse: (kinds, parameters [C, 8])."""
    k, p = pulse
    s = p[:, 2] / 5.0
    flat = p[:, 0] * _logistic(t, 6 * s, s) * (1.0 - _logistic(t, tau - 6 * s, s)) if 0 in k else None
    if flat is not None:
        return flat
    sr, sf, sm = p[:, 3] / 5.0, p[:, 4] / 5.0, p[:, 5] / 5.0
    return (p[:, 0] * _logistic(t, 6 * sr, sr) + (p[:, 1] - p[:, 0]) * _logistic(t, p[:, 2], sm)
            - p[:, 1] * _logistic(t, tau - 6 * sf, sf))


class _Bare:
    """H(t), jumps and readout of the bare-mode model on [T, Nt, Nr, Nf, M]."""

    def __init__(self, case, dims_of, theta, tau):
        self.tau, self.theta, self.rwa = tau, theta, case["frame"] == "rwa"
        self.kinds = [0] if case["M"] <= 8 else [1]
        pad = [max(d[i] if i < len(d) else 1 for d in dims_of) for i in range(3)]
        self.three, self.ro = len(dims_of[0]) == 3, 3 if len(dims_of[0]) == 3 else 2
        self.pad, self.lead = pad, 1
        idx = [torch.arange(n, dtype=torch.float64, device="cuda").reshape([-1 if i == k else 1 for i in range(3)]) for k, n in enumerate(pad)]
        self.mask = None
        if len(set(dims_of)) > 1:
            self.mask = torch.stack([((idx[0] < d[0]) & (idx[1] < d[1]) & (idx[2] < d[2])) for d in dims_of for _ in range(2)])[..., None]
        m = Model((1, 1))
        diag = m.wq * idx[0] + 0.5 * m.alpha * idx[0] * (idx[0] - 1) + m.wr * idx[1] + (m.wf * idx[2] if self.three else 0.0)
        self.diag, self.nexc, self.m = diag[None, ..., None], (idx[0] + idx[1] + idx[2])[None, ..., None], m
        self.damp = (-0.5 * (m.kappa * idx[self.ro - 1] + m.gamma * idx[0]))[None, ..., None]
        self.level = idx[0]

    def _drive(self, t):
        th = self.theta
        wd, phi = (th[:, 1], th[:, 3]) if self.kinds == [0] else (th[:, 6], th[:, 7])
        env = _envelope((self.kinds, th), self.tau, t)
        two = lambda v: v.repeat_interleave(2).reshape(-1, 1, 1, 1, 1)  # noqa: E731
        return two(env), two(wd), two(phi)

    def apply(self, z, t):
        """(-i H_eff z, [r z, b z], [kappa, gamma])."""
        env, wd, phi = self._drive(t)
        m, k = self.m, self.mask
        rz, bz = _shift(z, self.ro, False, k), _shift(z, 1, False, k)
        rd, bd = _shift(z, self.ro, True, k), _shift(z, 1, True, k)
        if self.rwa:
            h = (self.diag - wd * self.nexc) * z + m.g * (_shift(bd, 2, False, k) + _shift(bz, 2, True, k))
            if self.three:
                h = h + m.J * (_shift(rz, 2, True, k) + _shift(rd, 2, False, k))
            w = 0.5 * env * torch.exp(1j * phi)
            h = h + w * rz + w.conj() * rd
        else:
            x = bz + bd
            h = self.diag * z + m.g * (_shift(x, 2, False, k) + _shift(x, 2, True, k))
            y = rz + rd
            if self.three:
                h = h + m.J * (_shift(y, 2, False, k) + _shift(y, 2, True, k))
            h = h + env * torch.cos(wd * t + phi) * y
        return -1j * h + self.damp * z, [rz, bz], [m.kappa, m.gamma]

    def readout(self, z, t):
        return _shift(z, self.ro, False, self.mask)


class _Paper:
    """The normal-mode model of Sec. S2 in the frame of the drive, [T, Nl, Nu, Nt, M]."""

    def __init__(self, case, theta, tau):
        P = paper_params()
        self.pad = [int(x) for x in case["dims"].split("x")]
        nl, nu, nt = self.pad
        self.P, self.theta, self.tau, self.rot = P, theta, tau, case["frame"] == "rot"
        n = np.arange(-20, 21, dtype=float)
        e, v = np.linalg.eigh(np.diag(4.0 * P["Ec"] * n ** 2) - 0.5 * P["Ej"] * (np.eye(41, k=1) + np.eye(41, k=-1)))
        e = e[:nt]
        self.n1 = torch.tensor([abs(v[:, j] @ (n * v[:, j + 1])) for j in range(nt - 1)], dtype=torch.float64, device="cuda")
        wr, wf, J = P["wr"], P["wf"], P["J"]
        ev, vec = np.linalg.eig(np.array([[wr, J, 0, J], [J, wf, J, 0], [0, -J, -wr, -J], [-J, 0, -J, -wf]]))
        ev, vec = ev.real, vec.real
        x = []
        for i in np.argsort(ev)[2:]:
            y = vec[:, i] / math.sqrt(vec[0, i] ** 2 + vec[1, i] ** 2 - vec[2, i] ** 2 - vec[3, i] ** 2)
            x.append(y if y[1] > 0 else -y)
        (wl, wu), (cl, cu) = np.sort(ev)[2:], x
        part = lambda c: np.array([c[2], c[3], c[0], c[1]])  # noqa: E731
        S = np.linalg.inv(np.column_stack([part(cu), part(cl), cl, cu]).T)
        self.mu, self.nu, self.s = (S[0, 2] - S[0, 1], S[0, 3] - S[0, 0]), (S[1, 2] - S[1, 1], S[1, 3] - S[1, 0]), S[1]
        idx = [torch.arange(d, dtype=torch.float64, device="cuda").reshape([-1 if i == k else 1 for i in range(3)]) for k, d in enumerate(self.pad)]
        et = torch.tensor(e - e[0], dtype=torch.float64, device="cuda").reshape(1, 1, -1) - P["wd"] * idx[2]
        self.diag = ((wl - P["wd"]) * idx[0] + (wu - P["wd"]) * idx[1] + et)[None, ..., None]
        self.level, self.lead = idx[2], 2

    def _np(self, z):        # n_t^+ z and n_t^- z
        d = z.shape[3]
        w = self.n1.reshape(1, 1, 1, -1, 1)
        p, q = torch.zeros_like(z), torch.zeros_like(z)
        p.narrow(3, 0, d - 1).copy_(w * z.narrow(3, 1, d - 1))
        q.narrow(3, 1, d - 1).copy_(w * z.narrow(3, 0, d - 1))
        return p, q

    def readout(self, z, t, dag=False):
        s, ph = self.s, complex(np.exp(2j * self.P["wd"] * t)) if self.rot else 0.0
        if dag:
            ph = np.conj(ph)
        out = s[2] * _shift(z, 1, dag, None) + s[3] * _shift(z, 2, dag, None)
        if self.rot:
            out = out + ph * (s[0] * _shift(z, 2, not dag, None) + s[1] * _shift(z, 1, not dag, None))
        return out

    def apply(self, z, t):
        P = self.P
        env = _envelope(([0], self.theta), self.tau, torch.tensor(t, dtype=torch.float64, device="cuda"))
        if self.theta.shape[0] * 2 == z.shape[0]:
            env = env.repeat_interleave(2)
        env = env.reshape(-1, 1, 1, 1, 1)
        ph = complex(np.exp(2j * P["wd"] * t))
        h = self.diag * z
        zp, zm = self._np(z)
        for ax, mu, nu in ((1, self.mu[0], self.nu[0]), (2, self.mu[1], self.nu[1])):
            c, cd = _shift(z, ax, False, None), _shift(z, ax, True, None)
            h = h + 1j * P["g"] * mu * (_shift(zp, ax, True, None) - _shift(zm, ax, False, None))
            h = h - 0.5 * nu * env * (cd + c)
            if self.rot:
                h = h + 1j * P["g"] * mu * (ph * _shift(zm, ax, True, None) - np.conj(ph) * _shift(zp, ax, False, None))
                h = h + 0.5 * nu * env * (ph * cd + np.conj(ph) * c)
        f, b = self.readout(z, t), _shift(z, 3, False, None)
        damp = P["kappa"] * self.readout(f, t, dag=True) + P["gamma"] * _shift(b, 3, True, None)
        return -1j * h - 0.5 * damp, [f, b], [P["kappa"], P["gamma"]]


def _rhs(op, z, t, live):
    """Eq. S5 on z [T, N, M]; live [T, M] marks the columns a trajectory has."""
    T, N, M = z.shape
    five = [T] + op.pad + [M]
    a, ys, rates = op.apply(z.reshape(five), t)
    gram = z.mH @ z
    if live is not None:
        gram = gram + torch.diag_embed((~live).to(gram.dtype))
    chol = torch.linalg.cholesky(gram)
    out = a.reshape(T, N, M)
    for y, g in zip(ys, rates):
        y = y.reshape(T, N, M)
        x = torch.cholesky_solve(z.mH @ y, chol)
        out = out + 0.5 * g * (y @ x.mH)
    return out


def _rk4(f, z, t, dt):
    k1 = f(z, t)
    k2 = f(z + 0.5 * dt * k1, t + 0.5 * dt)
    k3 = f(z + 0.5 * dt * k2, t + 0.5 * dt)
    return z + (dt / 6.0) * (k1 + 2.0 * k2 + 2.0 * k3 + f(z + dt * k3, t + dt))


def _integrate(op, z, case, live=None):
    """Observables of the run and its final state."""
    dt, n, pe = case["dt"], case["steps"], case["pop_every"]
    T, N, M = z.shape
    nt = op.pad[0] if op.lead == 1 else op.pad[2]
    beta, pops, nphot = [], [], []
    for k in range(n + 1):
        r = op.readout(z.reshape([T] + op.pad + [M]), k * dt).reshape(T, N, M)
        beta.append((z.conj() * r).sum((1, 2)))
        if k % pe == 0:
            p = (z.abs() ** 2).sum(2).reshape([T] + op.pad)
            pops.append(p.sum((2, 3)) if op.lead == 1 else p.sum((1, 2)))
            nphot.append((r.abs() ** 2).sum((1, 2)))
        if k < n:
            z = _rk4(lambda y, t: _rhs(op, y, t, live), z, k * dt, dt)
    pops = torch.stack(pops, 1)
    return dict(beta=torch.stack(beta, 1), pops=pops.reshape(T, -1, nt), nphot=torch.stack(nphot, 1), trace=pops.sum(2)), z


def _losses(o, case, kappa, gamma):
    """(eps_a, T, Lambda) of Sec. S3.A and S3.B, trapezoids on the grids."""
    dt, n, pe = case["dt"], case["steps"], case["pop_every"]
    d = (o["beta"][1::2] - o["beta"][0::2]).abs() ** 2
    S = dt * (d.sum(1) - 0.5 * (d[:, 0] + d[:, -1]))
    eps = 0.5 * torch.erfc(0.5 * torch.sqrt(2.0 * ETA * kappa * S)) + 0.5 * n * dt * gamma
    hi = o["pops"][:, :, 2:].sum(2)
    hi = hi[0::2] + hi[1::2]
    ion = (hi.sum(1) - 0.5 * (hi[:, 0] + hi[:, -1])) * pe / n if hi.shape[1] > 1 else torch.zeros_like(eps)
    return eps, ion, torch.log10(eps + ion)


def _theta(case, seed, device="cuda"):
    th = torch.zeros(case["cands"], 8, dtype=torch.float64, device=device)
    for c, (_, p) in enumerate(_pulses(case, seed)):
        th[c, :len(p)] = torch.tensor(p, dtype=torch.float64)
    return th


def _host(o):
    return {k: v.detach().cpu() for k, v in o.items()}


def exact(case, seed):
    n, dt = case["steps"], case["dt"]
    tau = n * dt
    th = _theta(case, seed)
    stream_seed = torch.tensor(_signed(seed), dtype=torch.int64, device="cuda")
    if case["kind"] == "full":
        return _exact_full(case, th, tau)
    T = 2 * case["cands"]
    ts = _stream(stream_seed, torch.arange(T, dtype=torch.int64, device="cuda"))
    if case["kind"] == "sparse":
        op = _Paper(case, th, tau)
        z = _initial(op.pad, case["M"], ts, [0, 1] * case["cands"], 1)
        o, z = _integrate(op, z, case)
        P = paper_params()
        o["eps_a"], o["ion"], o["loss"] = _losses(o, case, P["kappa"], P["gamma"])
        if case["cands"] == 1:
            o["Z"] = z
        return _host(o)
    sizes = _sizes(case)
    op = _Bare(case, [d for d, _ in sizes], th, tau)
    if case["kind"] == "gradient":
        with torch.enable_grad():
            th = th.requires_grad_(True)
            op.theta = th
            z = _initial(op.pad, case["M"], ts, [0, 1] * case["cands"], op.pad[1] * op.pad[2])
            beta = []
            for k in range(n + 1):
                r = op.readout(z.reshape([T] + op.pad + [-1]), 0.0).reshape(z.shape)
                beta.append((z.conj() * r).sum((1, 2)))
                if k < n:
                    z = torch.utils.checkpoint.checkpoint(_rk4, lambda y, t: _rhs(op, y, t, None), z, k * dt, dt, use_reentrant=False)
            d = torch.stack(beta, 1)
            d = (d[1::2] - d[0::2]).abs() ** 2
            S = dt * (d.sum(1) - 0.5 * (d[:, 0] + d[:, -1]))
            eps = 0.5 * torch.erfc(0.5 * torch.sqrt(2.0 * ETA * KAPPA * S)) + 0.5 * tau * GAMMA
            w = torch.from_numpy(np.random.default_rng(seed).uniform(0.5, 1.5, case["cands"])).cuda()
            (eps * w).sum().backward()
        return _host({"eps_a": eps, "gradient": th.grad})
    live = None
    if case["kind"] == "resume":
        z = torch.from_numpy(_start_state(case, seed)).cuda()
    elif not case["uneven"]:
        z = _initial(op.pad, case["M"], ts, [0, 1] * case["cands"], op.pad[1] * op.pad[2])
    else:
        Mx = max(m for _, m in sizes)
        z = torch.zeros([T] + op.pad + [Mx], dtype=torch.complex128, device="cuda")
        live = torch.zeros(T, Mx, dtype=torch.bool, device="cuda")
        for c, (d, m) in enumerate(sizes):
            zc = _initial(d, m, ts[2 * c:2 * c + 2], [0, 1], d[1] * d[2])
            z[2 * c:2 * c + 2, :d[0], :d[1], :d[2], :m] = zc.reshape(2, *d, m)
            live[2 * c:2 * c + 2, :m] = True
        z = z.reshape(T, -1, Mx)
    o, z = _integrate(op, z, case, live)
    if case["uneven"]:     # the library's records are as wide as the largest level count of the batch
        o["pops"] = o["pops"][:, :, :max(d[0] for d, _ in sizes)]
    o["eps_a"], o["ionization"], o["loss"] = _losses(o, case, KAPPA, GAMMA)
    if case["cands"] == 1 and not case["uneven"]:
        o["Z"] = z
    return _host(o)


def _exact_full(case, th, tau):
    """Eq. 2 on the N x N density matrix from the pure state |0, 0, e>: with
    rho Hermitian, F = B + B^dag + sum_k L_k (L_k rho)^dag, B = -i H_eff rho."""
    op = _Paper(case, th, tau)
    N = int(np.prod(op.pad))
    rho = torch.zeros(1, N, N, dtype=torch.complex128, device="cuda")
    rho[0, 1, 1] = 1.0
    five = [1] + op.pad + [N]

    def f(r, t):
        a, ys, rates = op.apply(r.reshape(five), t)
        out = a.reshape(1, N, N)
        out = out + out.mH
        for i, (y, g) in enumerate(zip(ys, rates)):
            yd = y.reshape(1, N, N).mH.contiguous().reshape(five)
            ly = op.readout(yd, t) if i == 0 else _shift(yd, 3, False, None)
            out = out + g * ly.reshape(1, N, N)
        return out

    dt, n, pe, nt = case["dt"], case["steps"], case["pop_every"], op.pad[2]
    beta, pops, nphot = [], [], []
    for k in range(n + 1):
        fr = op.readout(rho.reshape(five), k * dt).reshape(1, N, N)
        beta.append(torch.diagonal(fr[0]).sum())
        if k % pe == 0:
            pops.append(torch.diagonal(rho[0]).real.reshape(-1, nt).sum(0))
            nphot.append(torch.diagonal(op.readout(fr.mH.contiguous().reshape(five), k * dt).reshape(N, N)).real.sum())
        if k < n:
            rho = _rk4(f, rho, k * dt, dt)
    pops = torch.stack(pops)
    return _host(dict(beta=torch.stack(beta), pops=pops, nphot=torch.stack(nphot), trace=pops.sum(1), rho=rho[0]))
