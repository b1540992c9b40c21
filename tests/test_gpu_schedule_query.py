"""The schedule that a context runs can be told: a run is, bit for bit, the run of the
schedule that the query names, and not that of the other."""
import math

import numpy as np
import pytest

import lr_inputs as li
from paper_2508_18114_gb300 import runner
from paper_2508_18114_gb300.sparse import SparseBatch, paper_model

pytestmark = pytest.mark.gpu


def _bare(cands):
    wl = li.c4(n_candidates=cands, n_steps=12)
    b = runner.make_batch(wl, precision="fp32_g64", engine="fused", pop_every=4, max_steps=12)
    b.set_initial(wl.init_seed, wl.eps)
    b.integrate(wl.dt, 12)
    z, wide = b.get_state(0), b.wide
    b.close()
    return z, wide


def _sparse(T):
    tp = 2 * math.pi
    model = paper_model(100, 4, 5, frame="rot", Ec=tp * 0.315, Ej=51 * tp * 0.315, wr=tp * 7.2, wf=tp * 7.21,
                        g=tp * 0.15, J=tp * 0.03, kappa=tp * 0.03, gamma=tp * 8e-6, wd=tp * 7.18)
    b = SparseBatch(model, 20, [(0, (1.5, tp * 7.18, 0.004, 0.0))] * T, 0.02, 12, precision="fp32_g64")
    assert b.fused
    b.set_initial([i % 2 for i in range(T)], 7, 1e-4)
    b.integrate(5e-4, 12)
    return b.get_state()[0], b.wide


@pytest.mark.parametrize("run,var,n,wide", [(_bare, "LR_FUSED_WIDE", 1, True), (_bare, "LR_FUSED_WIDE", 8, False),
                                            (_sparse, "LR_SPARSE_WIDE", 2, True), (_sparse, "LR_SPARSE_WIDE", 40, False)])
def test_the_query_names_the_schedule_that_runs(monkeypatch, run, var, n, wide):
    monkeypatch.delenv(var, raising=False)
    z, w = run(n)
    assert w == wide
    forced = {}
    for v in ("0", "1"):
        monkeypatch.setenv(var, v)
        forced[v], w = run(n)
        assert w == (v == "1")
    assert np.array_equal(z, forced["1" if wide else "0"])
    assert not np.array_equal(z, forced["0" if wide else "1"])


def test_engines_without_a_choice():
    wl = li.c1(n_steps=4)
    b = runner.make_batch(wl, precision="fp64", engine="plain", max_steps=4)
    assert not b.wide
    b.close()
