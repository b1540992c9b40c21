"""The wide schedule of batches that are far smaller than the GPU (a few
launches per RK4 stage over the whole chip, LR_FUSED_WIDE / LR_SPARSE_WIDE)
against the FP64 engines, and its CUDA graph replays against direct calls.

Tolerance: a stage rounds every entry of the state a few times (at most 8, u =
2^-24 each) and the roundings add up like a random walk over the 4 S stages:
8 u sqrt(4 S) of the state's norm, 6e-6 at S = 40; the signal and the
populations are quadratic in the state, with |r| <= sqrt(N_f): twice that
times 5.
"""
import math

import numpy as np
import pytest

import lr_inputs as li
from paper_2508_18114_gb300 import LrError, runner
from paper_2508_18114_gb300.sparse import SparseBatch, paper_model

pytestmark = pytest.mark.gpu

STEPS = 40
TOL = 8 * 2.0 ** -24 * math.sqrt(4 * STEPS)


def _workload(dims, ranks, kind, frame="lab"):
    cands = []
    for k, M in enumerate(ranks):
        m = li.ModelParams(dims=dims[k % len(dims)], wq=37.7, alpha=-1.9, wr=47.1, g=0.94, kappa=0.31, gamma=2e-3,
                           **({"wf": 47.2, "J": 0.63} if len(dims[k % len(dims)]) == 3 else {}))
        p = (2.0, 47.0, 0.01, 0.3) if kind == 0 else (2.0, 1.2, 0.01, 0.004, 0.004, 0.004, 47.0, 0.3)
        cands.append(li.Candidate(m, M, li.PulseParams(kind, p)))
    return li.Workload("wide", cands, 5e-4, STEPS, STEPS * 5e-4, init_seed=5, eps=1e-4,
                       frame=frame)


def _run(wl, precision, engine):
    b = runner.make_batch(wl, precision=precision, engine=engine, pop_every=8, max_steps=STEPS)
    b.set_initial(wl.init_seed, wl.eps)
    b.integrate(wl.dt, 13)
    b.integrate(wl.dt, STEPS - 13)
    o = b.observables()
    z = [b.get_state(j) for j in range(b.n_traj)]
    b.close()
    return o, z


@pytest.mark.parametrize("dims,ranks,frame", [
    ([(3, 5, 3)], [1], "lab"),                       # a single column: no pair to share a thread
    ([(4, 9)], [7], "lab"),                          # two modes, odd rank, fewer rows than a block
    ([(3, 7, 5), (2, 16, 4)], [31, 2, 8], "lab"),    # uneven ranks and sizes
    ([(10, 20, 10)], [20], "lab"),                   # the size that takes the schedule by itself
    ([(5, 11, 6)], [32, 32], "rwa"),                 # the largest rank, rotating frame
])
def test_wide_against_fp64(monkeypatch, dims, ranks, frame):
    wl = _workload(dims, ranks, 0 if len(ranks) == 1 else 1, frame)
    monkeypatch.setenv("LR_FUSED_WIDE", "1")
    o32, z32 = _run(wl, "fp32_g64", "fused")
    w64, y64 = _run(wl, "fp64", "fused")
    monkeypatch.delenv("LR_FUSED_WIDE")
    o64, z64 = _run(wl, "fp64", "plain")
    # FP64: the plain engine's kernels and arithmetic, to the last bit
    assert all(np.array_equal(a, b) for a, b in zip(y64, z64))
    assert all(np.array_equal(w64[k], o64[k]) for k in ("beta", "pops", "nphot", "trace", "eps_a"))
    for a, b in zip(z32, z64):
        assert np.linalg.norm(a - b) <= TOL * np.linalg.norm(b)
    for k in ("beta", "pops", "nphot", "trace"):
        assert np.abs(o32[k] - o64[k]).max() <= 10 * TOL * max(1.0, np.abs(o64[k]).max()), k


def test_wide_graph_replays(monkeypatch):
    """Replays continue the run bit by bit; one past max_steps runs nothing."""
    monkeypatch.setenv("LR_FUSED_WIDE", "1")
    wl = _workload([(3, 7, 5)], [6], 1)
    want, zw = _run(wl, "fp32_g64", "fused")
    b = runner.make_batch(wl, precision="fp32_g64", engine="fused", pop_every=8, max_steps=STEPS)
    b.set_initial(wl.init_seed, wl.eps)
    g = b.capture_integrate(wl.dt, STEPS // 4)
    for _ in range(4):
        g.replay()
    b.sync()
    got = b.observables()
    for k in ("beta", "pops", "nphot", "trace", "eps_a"):
        assert np.array_equal(got[k], want[k]), k
    g.replay()
    with pytest.raises(LrError) as ei:
        b.sync()
    assert ei.value.status == 8
    assert np.array_equal(b.get_state(0), zw[0])
    b.close()


@pytest.mark.parametrize("dims,M,T", [((8, 2, 3), 1, 2), ((9, 3, 4), 13, 3), ((20, 4, 5), 20, 2), ((12, 3, 5), 32, 1)])
def test_sparse_wide_against_fp64(monkeypatch, dims, M, T):
    tp = 2 * math.pi
    model = paper_model(*dims, frame="rot", Ec=tp * 0.315, Ej=51 * tp * 0.315, wr=tp * 7.2, wf=tp * 7.21, g=tp * 0.15,
                        J=tp * 0.03, kappa=tp * 0.03, gamma=tp * 8e-6, wd=tp * 7.18)
    out = {}
    for prec, wide in (("fp64", "0"), ("fp32_g64", "1")):
        monkeypatch.setenv("LR_SPARSE_WIDE", wide)
        b = SparseBatch(model, M, [(0, (1.5, tp * 7.18, 0.004, 0.0))] * T, STEPS * 5e-4, STEPS, pop_every=8, precision=prec)
        b.set_initial([i % 2 for i in range(T)], 7, 1e-4)
        b.integrate(5e-4, 13)
        b.integrate(5e-4, STEPS - 13)
        out[prec] = (b.observables(), b.get_state())
    (o32, z32), (o64, z64) = out["fp32_g64"], out["fp64"]
    assert np.linalg.norm(z32 - z64) <= TOL * np.linalg.norm(z64)
    for k in ("beta", "pops", "nphot", "trace"):
        assert np.abs(o32[k] - o64[k]).max() <= 10 * TOL * max(1.0, np.abs(o64[k]).max()), k
