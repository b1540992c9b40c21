"""Assignment of an uneven batch to the fused engine's teams: every trajectory
runs once, whichever team takes it, and its result does not depend on the rest
of the batch (the arithmetic of a trajectory is the plan's, not the batch's)."""
import numpy as np
import pytest

import lr_inputs as li
from paper_2508_18114_gb300 import runner

pytestmark = pytest.mark.gpu


def _candidate(k):
    dims = [(3, 5, 3), (2, 9, 4), (4, 6, 5), (2, 4, 3)][k % 4]
    m = li.ModelParams(dims=dims, wq=37.7, alpha=-1.9, wr=47.1, g=0.94, kappa=0.31, gamma=2e-3, wf=47.2, J=0.63)
    return li.Candidate(m, 1 + (7 * k) % 11, li.PulseParams(0, (2.0 + 0.01 * k, 47.0, 0.01, 0.3)))


def _run(ks):
    wl = li.Workload("teams", [_candidate(k) for k in ks], 5e-4, 20, 0.01, init_seed=5, eps=1e-4)
    b = runner.make_batch(wl, precision="fp64", engine="fused", pop_every=10, max_steps=20)
    for j, k in enumerate(ks):   # a state of the candidate's own, not of its place in the batch
        N, M = int(np.prod(_candidate(k).model.dims)), _candidate(k).M
        g = np.random.default_rng(k)
        for lvl in range(2):
            q = np.linalg.qr(g.standard_normal((N, M)) + 1j * g.standard_normal((N, M)))[0]
            b.set_state(2 * j + lvl, q * 10.0 ** -(0.2 * np.arange(M)), 0)
    b.integrate(wl.dt, 20)
    z = [b.get_state(j) for j in range(2 * len(ks))]
    o = b.observables()
    b.close()
    return z, o


@pytest.mark.parametrize("team,n", [(1, 90), (1, 160), (2, 60), (4, 3)])
def test_uneven_batch_equals_its_parts(monkeypatch, team, n):
    monkeypatch.setenv("LR_FUSED_C", str(team))
    z, o = _run(range(n))
    for part in ([0, 1, 2, 3, 12], [n - 1, n // 2, 9 % n, 10 % n]):   # ranks up to 11 in both: the same padded rank
        part = [k for k in part if k < n]
        zp, op = _run(part + [8, 3])
        for j, k in enumerate(part):
            for lvl in range(2):
                assert np.array_equal(zp[2 * j + lvl], z[2 * k + lvl]), (k, lvl)
                assert np.array_equal(op["beta"][2 * j + lvl], o["beta"][2 * k + lvl])
