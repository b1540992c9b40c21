"""The fixed-rank initial state on the device against the oracle's Householder
QR, at the edges of its row tiles (128), of a team's row split and of the rank.

The q_j agree up to a phase per column, fixed here by the sign of the diagonal
of R: both are the columns of one QR factorisation, so column j differs by the
phase of <q_j, q_j'>. FP64 bound: both sides are orthonormal to a few 2^-53 per
entry and the draws differ by a few ulp, amplified by cond(W) <= 1e3 at M = N;
1e-11 absolute. FP32: the entries rounded once, 2^-24 of the largest (1).
"""
import numpy as np
import pytest

import lr_inputs as li
from oracle import init_state

pytestmark = pytest.mark.gpu

EPS, SEED = 1e-3, 77


def _model(dims):
    p = li.c1().candidates[0].model if len(dims) == 2 else li.c2().candidates[0].model
    import dataclasses
    return dataclasses.replace(p, dims=dims)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("fp32_g64", 1.3e-7)])
@pytest.mark.parametrize("cands", [
    [((2, 4), 8)],                                     # M = N: square Gaussian factor, two rounds
    [((4, 10), 1)],                                    # no padding columns
    [((4, 32), 32), ((3, 43), 20), ((4, 10), 2)],      # 128, 129 and 40 rows, uneven ranks
    [((5, 17, 3), 13)],                                # 255 rows split over a team
    [((10, 20, 10), 20)],                              # 2000 rows, 8 CTAs
    [((4, 33), 5)] * 80,                               # more trajectories than SMs: one CTA each
])
def test_initial_state_equals_the_oracle(precision, tol, cands):
    from paper_2508_18114_gb300 import LowRankBatch
    b = LowRankBatch([_model(d) for d, _ in cands], [m for _, m in cands], precision=precision, max_steps=2)
    b.set_pulse([(0, (0.1, 47.0, 1.0, 0.0))] * len(cands), 10.0)
    b.set_initial(SEED, EPS)
    picked = range(2 * len(cands)) if len(cands) < 10 else (0, 1, 81, 159)
    for tj in picked:
        dims, M = cands[tj // 2]
        N = int(np.prod(dims))
        want = init_state.initial_state(N, M, (tj % 2) * (N // dims[0]), EPS, SEED, tj)
        got = b.get_state(tj)
        ph = np.sum(want.conj() * got, axis=0)
        got = got * (ph.conj() / np.abs(ph))
        assert np.abs(got - want).max() < tol
