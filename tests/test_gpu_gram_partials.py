"""A team of CTAs adds its Gram partials of an FP32 state in FP64.

One column with the entries 1 (rows of the first CTA) and x (rows of the last):
both partials, 1 and x^2, are exact, and x is chosen so that the low float of x^2
lies below 2^-24 of the high one. A double-word sum with 1 drops it (2^-50.1 of
the sum); FP64 rounds once (2^-53), and the recorded eigenvalue is that sum.
"""
import math

import numpy as np
import pytest

import lr_inputs as li
from paper_2508_18114_gb300 import runner

pytestmark = pytest.mark.gpu


def _x():
    """An FP32 number near 2^-13 whose square is almost half way between two FP32 numbers."""
    for k in range(1, 10000):
        x = float(np.float32(2.0 ** -13 * (1 + k * 2.0 ** -23)))
        p = float(np.float32(x * x))   # x * x is exact in FP64
        if x * x - p > 0.93 * 2.0 ** -50:
            return x
    raise AssertionError("no such x")


@pytest.mark.parametrize("team", [2, 4, 8])
def test_partials_of_a_team_are_added_in_fp64(monkeypatch, team):
    monkeypatch.setenv("LR_FUSED_C", str(team))
    dims, x = (3, 8, 3), _x()
    m = li.ModelParams(dims=dims, wq=37.7, alpha=-1.9, wr=47.1, g=0.94, kappa=0.31, gamma=2e-3, wf=47.2, J=0.63)
    wl = li.Workload("gram", [li.Candidate(m, 1, li.PulseParams(0, (1.0, 47.0, 0.01, 0.3)))], 5e-4, 4, 0.01,
                     init_seed=5, eps=1e-4)
    b = runner.make_batch(wl, precision="fp32_g64", engine="fused", pop_every=1, max_steps=4, record_gram=True)
    assert b.query().team_size == team
    z = np.zeros((72, 1), complex)
    z[0, 0] = 1.0            # resonator level 0: the first CTA
    z[7 * 3, 0] = x          # resonator level 7: the last
    for j in (0, 1):
        b.set_state(j, z, 0)
    b.integrate(wl.dt, 0)
    _, eig = b.diagnostics()
    b.close()
    for j in (0, 1):
        assert abs(math.fsum([eig[j, 0, 0], -1.0, -x * x])) <= 2.0 ** -52
