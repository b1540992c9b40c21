"""lr_backward runs in the workspace that its memory formula states, and a workspace with
room for a segment's stage inputs gives the same gradient."""
import ctypes as C

import numpy as np
import pytest
import torch

import lr_inputs as li
from paper_2508_18114_gb300 import runner

pytestmark = pytest.mark.gpu

S = 24


def _batch(precision):
    m = li.ModelParams(dims=(4, 9, 5), wq=37.7, alpha=-1.9, wr=47.1, g=0.94, kappa=0.31, gamma=2e-3, wf=47.2, J=0.63)
    p = li.PulseParams(1, (2.0, 1.2, 0.006, 0.003, 0.003, 0.003, 47.0, 0.3))
    wl = li.Workload("bwd", [li.Candidate(m, 7, p)] * 40, 5e-4, S, S * 5e-4, init_seed=5, eps=1e-4)
    b = runner.make_batch(wl, precision=precision, engine="auto", pop_every=8, max_steps=S)
    b.set_initial(wl.init_seed, wl.eps)
    b.integrate(wl.dt, S)
    return b


@pytest.mark.parametrize("precision", ["fp64", "fp32_g64"])
@pytest.mark.parametrize("K", [5, 24, 200])
def test_workspace_as_stated_and_kept_stages_give_one_gradient(monkeypatch, precision, K):
    b = _batch(precision)
    sz = C.c_size_t()
    assert b._lib.lr_backward_workspace_size(b._h, K, C.byref(sz)) == 0
    T = 80 * 180 * 7 * (16 if precision == "fp64" else 8)   # the states of 80 trajectories
    # tables: partial sums of 12 row blocks (twice), 16 M x M factors of rank 32, beta, drive
    tables = 80 * (2 * 12 * 8 * (6 * 49 + 20) + 16 * 1024 * 16 + 16 * (S + 1) + 8 * 12 * 200)
    assert sz.value <= (-(-S // K) + K + 15) * T + tables
    w = np.linspace(0.5, 1.5, 40)
    kept = b.backward(w, ckpt_every=K)
    assert np.array_equal(b.backward(w, ckpt_every=K, keep=False), kept)
    # a device without the memory for the kept stages: the stated workspace is taken
    empty, tried = torch.empty, []

    def small(n, *a, **k):
        tried.append(n)
        if n > sz.value + 256:
            raise torch.cuda.OutOfMemoryError("no memory")
        return empty(n, *a, **k)

    monkeypatch.setattr(torch, "empty", small)
    assert np.array_equal(b.backward(w, ckpt_every=K), kept)
    assert tried[-1] == sz.value + 256 and tried[0] > tried[-1]
    monkeypatch.undo()
    b.close()
