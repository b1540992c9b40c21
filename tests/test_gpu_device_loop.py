"""A long direct call of the wide schedule is one device-side loop: the same bits as short
calls, which are launched step by step, and the host does not wait for it."""
import math
import time

import numpy as np
import pytest
import torch

import lr_inputs as li
from paper_2508_18114_gb300 import runner
from paper_2508_18114_gb300.sparse import SparseBatch, paper_model

pytestmark = pytest.mark.gpu

S = 203    # no multiple of the body's steps, of pop_every or of a channel table
TP = 2 * math.pi


def _bare(precision, max_steps=S, dims=None):
    wl = li.c4(n_candidates=1, n_steps=max_steps)
    b = runner.make_batch(wl, precision=precision, engine="fused", pop_every=7, max_steps=max_steps)
    b.set_initial(wl.init_seed, wl.eps)
    return b


def _sparse(precision, max_steps=S):
    model = paper_model(40, 3, 4, frame="rot", Ec=TP * 0.315, Ej=51 * TP * 0.315, wr=TP * 7.2, wf=TP * 7.21,
                        g=TP * 0.15, J=TP * 0.03, kappa=TP * 0.03, gamma=TP * 8e-6, wd=TP * 7.18)
    b = SparseBatch(model, 28, [(0, (1.5, TP * 7.18, 0.004, 0.0))] * 2, max_steps * 5e-4, max_steps, pop_every=7,
                    precision=precision)
    b.set_initial([0, 1], 7, 1e-4)
    return b


def _result(b):
    o = b.observables()
    z = b.get_state() if isinstance(b, SparseBatch) else np.stack([b.get_state(j) for j in (0, 1)])
    return [z] + [o[k] for k in ("beta", "pops", "nphot", "trace")]


CASES = [(_bare, "fp32_g64"), (_bare, "fp64"), (_sparse, "fp32_g64")]


@pytest.mark.parametrize("make,precision", CASES)
def test_loop_equals_short_calls(monkeypatch, make, precision):
    for k in ("LR_FUSED_WIDE", "LR_SPARSE_WIDE"):
        monkeypatch.setenv(k, "1")
    a, b = make(precision), make(precision)
    a.integrate(5e-4, S)
    for n in (13, *[20] * 9, 10):
        b.integrate(5e-4, n)
    for x, y in zip(_result(a), _result(b)):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("make,precision", CASES)
def test_host_and_other_streams_go_on(monkeypatch, make, precision):
    """Two contexts on two streams: both calls return before a quarter of the run has
    passed, and both results are those of a context alone."""
    for k in ("LR_FUSED_WIDE", "LR_SPARSE_WIDE"):
        monkeypatch.setenv(k, "1")
    n = 1000
    alone = make(precision, n)
    alone.integrate(5e-4, n)
    want = _result(alone)
    streams = [torch.cuda.Stream() for _ in range(2)]
    batches = [make(precision, n) for _ in streams]
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for b, s in zip(batches, streams):
        b.integrate(5e-4, n, stream=s)
    t1 = time.perf_counter()
    torch.cuda.synchronize()
    t2 = time.perf_counter()
    for b in batches:
        for x, y in zip(_result(b), want):
            assert np.array_equal(x, y)
    assert t1 - t0 < 0.25 * (t2 - t0)


def test_more_step_sizes_than_kept_graphs(monkeypatch):
    """A context keeps four graphs; a fifth (dt, tau) takes the place of the oldest."""
    monkeypatch.setenv("LR_FUSED_WIDE", "1")
    wl = li.c4(n_candidates=1, n_steps=80)
    pulses = [(c.pulse.kind, c.pulse.p) for c in wl.candidates]
    b = runner.make_batch(wl, precision="fp32_g64", engine="fused", pop_every=7, max_steps=80)
    first = []
    for turn in range(2):
        for k in range(6):
            b.set_pulse(pulses, wl.tau * (1 + k // 3))
            b.set_initial(wl.init_seed, wl.eps)
            b.integrate(wl.dt * (1 + k % 3), 80)
            r = _result(b)
            if turn == 0:
                first.append(r)
                assert k == 0 or not np.array_equal(r[0], first[k - 1][0])
            else:
                assert all(np.array_equal(x, y) for x, y in zip(r, first[k]))
    b.close()
