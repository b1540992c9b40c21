"""The persistent kernels (teams of CTAs) on batches that take the wide schedule by
themselves: the tests that are meant for those kernels, run with the wide schedule off,
and the sparse kernel at the ranks where its M x M phase changes layout.
"""
import math

import numpy as np
import pytest

from paper_2508_18114_gb300 import LowRankBatch, LrError
from paper_2508_18114_gb300.sparse import SparseBatch, paper_model

from test_gpu_diagnostics import test_spectrum_and_purity_match_oracle  # noqa: F401
from test_gpu_fused import (test_c2_full_size_fp64_and_fp32, test_fused_not_positive_definite_is_reported,  # noqa: F401
                            test_fused_resume_is_bitwise)
from test_gpu_full_pulse import test_paper_model_full_pulse_sparse  # noqa: F401
from test_gpu_mm_phase import test_ranks_at_the_edges_of_the_sweep  # noqa: F401
from test_gpu_paper_model import test_fused_team_default_for_small_batches, test_large_rank  # noqa: F401
from test_gpu_rwa import test_rwa_three_modes_match_oracle  # noqa: F401

pytestmark = pytest.mark.gpu

TP = 2 * math.pi
STEPS = 40
# 8 roundings of 2^-24 per entry and stage, a random walk over 4 STEPS stages
TOL = 8 * 2.0 ** -24 * math.sqrt(4 * STEPS)


@pytest.fixture(autouse=True)
def teams(monkeypatch):
    """No wide schedule, and every run is checked for it."""
    monkeypatch.setenv("LR_FUSED_WIDE", "0")
    monkeypatch.setenv("LR_SPARSE_WIDE", "0")
    for cls in (LowRankBatch, SparseBatch):
        def checked(self, *a, _run=cls.integrate, **k):
            assert not self.wide
            return _run(self, *a, **k)
        monkeypatch.setattr(cls, "integrate", checked)


def _sparse(M, T, precision):
    model = paper_model(9, 3, 4, frame="rot", Ec=TP * 0.315, Ej=51 * TP * 0.315, wr=TP * 7.2, wf=TP * 7.21, g=TP * 0.15,
                        J=TP * 0.03, kappa=TP * 0.03, gamma=TP * 8e-6, wd=TP * 7.18)
    b = SparseBatch(model, M, [(0, (1.5, TP * 7.18, 0.004, 0.0))] * T, STEPS * 5e-4, STEPS, pop_every=8,
                    precision=precision)
    b.set_initial([i % 2 for i in range(T)], 7, 1e-4)
    return b


@pytest.mark.parametrize("team", [1, 3])
@pytest.mark.parametrize("M", [1, 8, 22, 31, 32])
def test_sparse_kernel_at_the_edges_of_the_sweep(monkeypatch, M, team):
    """One entry, two warps, half the warps, every warp, more entries than threads."""
    monkeypatch.setenv("LR_SPARSE_C", str(team))
    out = []
    for precision in ("fp64", "fp32_g64"):
        b = _sparse(M, 2, precision)
        assert precision == "fp64" or b.team == team
        b.integrate(5e-4, 13)     # the table of channel factors ends within both calls
        b.integrate(5e-4, STEPS - 13)
        out.append((b.observables(), b.get_state()))
    (o64, z64), (o32, z32) = out
    assert np.linalg.norm(z32 - z64) <= TOL * np.linalg.norm(z64)
    for k in ("beta", "pops", "nphot", "trace"):
        assert np.abs(o32[k] - o64[k]).max() <= 10 * TOL * max(1.0, np.abs(o64[k]).max()), k


@pytest.mark.parametrize("team", [1, 3])
@pytest.mark.parametrize("M", [5, 32])
def test_sparse_kernel_reports_equal_columns(monkeypatch, M, team):
    monkeypatch.setenv("LR_SPARSE_C", str(team))
    b = _sparse(M, 2, "fp32_g64")
    z = b.get_state()
    z[1, :, M - 1] = z[1, :, 0]
    b.set_state(z, 0)
    b.integrate(5e-4, 3)
    with pytest.raises(LrError) as ei:
        b.observables()
    assert ei.value.status == 5
