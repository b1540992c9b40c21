"""The initial state of a trajectory does not depend on the batch around it: neither on
the SMs that the batch leaves to it (teams of 8, 3 or 1 CTAs) nor on the other
candidates' sizes (M = N asks for a second orthonormalisation round)."""
import dataclasses

import numpy as np
import pytest

import lr_inputs as li
from paper_2508_18114_gb300 import LowRankBatch

pytestmark = pytest.mark.gpu


def _states(cands, precision):
    base = {2: li.c1().candidates[0].model, 3: li.c2().candidates[0].model}
    b = LowRankBatch([dataclasses.replace(base[len(d)], dims=d) for d, _ in cands], [m for _, m in cands],
                     precision=precision, max_steps=2)
    b.set_pulse([(0, (0.1, 47.0, 1.0, 0.0))] * len(cands), 10.0)
    b.set_initial(77, 1e-3)
    z = [b.get_state(j) for j in (0, 1)]
    b.close()
    return z


@pytest.mark.parametrize("precision", ["fp64", "fp32_g64"])
@pytest.mark.parametrize("cand", [((10, 20, 10), 20), ((4, 33), 5), ((5, 17, 7), 32), ((3, 7), 4)])
def test_initial_state_is_the_trajectorys_own(precision, cand):
    alone = _states([cand], precision)
    for others in ([((2, 4), 8)] * 2, [((4, 10), 3)] * 24, [((2, 4), 8), ((3, 43), 30)] * 80):
        for a, b in zip(alone, _states([cand] + others, precision)):
            assert np.array_equal(a, b), len(others)
