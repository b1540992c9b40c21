"""Stream capture of small batches: a graph of the teams' kernel, whatever the number of
steps, also where a direct call takes the whole-chip launches; direct calls and replays
continue one another.

Tolerance of a run that mixes the schedules: 8 roundings of u = 2^-24 per entry and
stage, adding up like a random walk over the 4 S stages.
"""
import ctypes as C
import math

import numpy as np
import pytest
import torch

import lr_inputs as li
from paper_2508_18114_gb300 import runner
from paper_2508_18114_gb300.sparse import SparseBatch, paper_model

pytestmark = pytest.mark.gpu

N1 = 10


def _captured(call):
    """(graph, nodes) of call(stream) captured on a stream of its own."""
    cu = C.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph, n = C.c_void_p(), C.c_size_t()
    assert cu.cuStreamBeginCapture_v2(C.c_void_p(st.cuda_stream), 1) == 0
    call(st)
    assert cu.cuStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    return cu, graph, n.value


def _replay(cu, graph, times):
    ex = C.c_void_p()
    assert cu.cuGraphInstantiateWithFlags(C.byref(ex), graph, C.c_ulonglong(0)) == 0
    for _ in range(times):
        assert cu.cuGraphLaunch(ex, C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert cu.cuGraphExecDestroy(ex) == 0 and cu.cuGraphDestroy(graph) == 0


@pytest.mark.parametrize("precision", ["fp32_g64", "fp64"])
def test_capture_of_a_small_batch_is_three_kernels(monkeypatch, precision):
    wl = li.c4(n_candidates=1, n_steps=4 * N1)
    monkeypatch.delenv("LR_FUSED_WIDE", raising=False)
    b = runner.make_batch(wl, precision=precision, engine="fused", pop_every=5, max_steps=4 * N1)
    b.set_initial(wl.init_seed, wl.eps)
    b.integrate(wl.dt, N1)
    start = [b.get_state(j) for j in (0, 1)]
    cu, graph, nodes = _captured(lambda st: b.integrate(wl.dt, N1, stream=st))
    assert nodes <= 3
    b.sync()
    _replay(cu, graph, 2)
    b.sync()
    assert b.query().step == 3 * N1
    got, ob = [b.get_state(j) for j in (0, 1)], b.observables()
    b.integrate(wl.dt, N1)
    after = b.get_state(0)
    b.close()
    monkeypatch.setenv("LR_FUSED_WIDE", "0")
    b = runner.make_batch(wl, precision=precision, engine="fused", pop_every=5, max_steps=4 * N1)
    for j in (0, 1):
        b.set_state(j, start[j], N1)
    b.integrate(wl.dt, 2 * N1)
    for j in (0, 1):
        assert np.array_equal(b.get_state(j), got[j])
    assert np.array_equal(b.observables()["beta"][:, N1:3 * N1 + 1], ob["beta"][:, N1:3 * N1 + 1])
    b.integrate(wl.dt, N1)
    assert np.linalg.norm(b.get_state(0) - after) <= 8 * 2.0 ** -24 * math.sqrt(4 * N1)
    b.close()


def test_sparse_capture_is_the_fused_kernel(monkeypatch):
    tp = 2 * math.pi
    model = paper_model(40, 3, 4, frame="rot", Ec=tp * 0.315, Ej=51 * tp * 0.315, wr=tp * 7.2, wf=tp * 7.21,
                        g=tp * 0.15, J=tp * 0.03, kappa=tp * 0.03, gamma=tp * 8e-6, wd=tp * 7.18)
    z = {}
    for wide in ("", "0"):
        if wide:
            monkeypatch.setenv("LR_SPARSE_WIDE", wide)
        else:
            monkeypatch.delenv("LR_SPARSE_WIDE", raising=False)
        b = SparseBatch(model, 28, [(0, (1.5, tp * 7.18, 0.004, 0.0))] * 2, 0.02, 3 * N1, pop_every=5,
                        precision="fp32_g64")
        b.set_initial([0, 1], 7, 1e-4)
        b.integrate(5e-4, N1)
        cu, graph, nodes = _captured(lambda st: b.integrate(5e-4, N1, stream=st))
        assert nodes <= 2
        _replay(cu, graph, 1)
        b.integrate(5e-4, N1)
        b.observables()
        z[wide] = b.get_state()
    assert np.linalg.norm(z[""] - z["0"]) <= 8 * 2.0 ** -24 * math.sqrt(12 * N1) * np.linalg.norm(z["0"])
