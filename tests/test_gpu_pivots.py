"""The limits of a pivot below which a state is refused (LR_ERR_NOT_PD).

Two columns e_a and e_a + d e_b: the second pivot is d^2, its diagonal entry 1 + d^2.
The rows a and b are annihilated by both jump operators and the step is 2^-20, so the
Gram matrix stays that one to 1e-11 d^2 or its rounding.
"""
import numpy as np
import pytest

import lr_inputs as li
from paper_2508_18114_gb300 import LrError, runner
from paper_2508_18114_gb300.sparse import SparseBatch

pytestmark = pytest.mark.gpu

H = 2.0 ** -20


def _bare(z, engine):
    m = li.ModelParams(dims=(3, 6, 4), wq=0.2, alpha=-0.1, wr=0.3, g=0.1, kappa=1e-3, gamma=1e-3, wf=0.25, J=0.1)
    wl = li.Workload("pivot", [li.Candidate(m, z.shape[1], li.PulseParams(0, (0.0, 0.3, 0.01, 0.0)))], H, 1, 1.0,
                     init_seed=1, eps=1e-4)
    b = runner.make_batch(wl, precision="fp64", engine=engine, pop_every=1, max_steps=1)
    for j in (0, 1):
        b.set_state(j, z, 0)
    b.integrate(H, 1)
    return b


def _sparse(z):
    N = z.shape[0]
    n = np.arange(N)
    val = np.zeros((3 * N, 2))
    val[:N, 1] = -0.25
    val[N:, 0] = 2.0 ** -10
    model = dict(N=N, nnz=3 * N, n_jumps=1, n_levels=2, wd=1.0, chan=np.full(3 * N, 2), level=n % 2,
                 rowptr=np.concatenate([o * N + np.arange(N + 1) for o in range(3)]), col=np.concatenate([n, n, n]),
                 val=val.reshape(-1))
    b = SparseBatch(model, z.shape[1], [(0, (1.0, 1.0, 0.01, 0.0))] * 2, 1.0, 1, precision="fp64")
    b.set_state(np.stack([z, z]), 0)
    b.integrate(H, 1)
    return b


def _refused(b):
    try:
        b.observables()
    except LrError as e:
        assert e.status == 5
        return True
    return False


def _pair(d2):
    z = np.zeros((72, 2), complex)
    z[0, 0] = z[0, 1] = 1.0
    z[8, 1] = np.sqrt(d2)      # resonator level 2, transmon and filter in their ground states
    return z


@pytest.mark.parametrize("d2,refused", [(4e-15, False), (1.3e-14, False), (0.0, True)])
def test_fp64_launches_refuse_only_what_rounding_leaves(d2, refused):
    assert _refused(_bare(_pair(d2), "plain")) == refused
    assert _refused(_sparse(_pair(d2))) == refused


@pytest.mark.parametrize("M", [2, 9, 32])
def test_equal_columns_are_refused(M):
    g = np.random.default_rng(M)
    z = (g.standard_normal((72, M)) + 1j * g.standard_normal((72, M))) * 10.0 ** -np.linspace(0, 3, M)
    z[:, M - 1] = z[:, 0]
    assert _refused(_bare(z, "plain"))
    assert _refused(_sparse(z))


@pytest.mark.parametrize("wide", ["0", "1"])
@pytest.mark.parametrize("d2,refused", [(2e-13, False), (5e-14, True)])
def test_a_fused_context_refuses_the_same_in_either_schedule(monkeypatch, d2, refused, wide):
    monkeypatch.setenv("LR_FUSED_WIDE", wide)
    assert _refused(_bare(_pair(d2), "fused")) == refused
