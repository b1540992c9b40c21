"""The M x M phase of the fused kernels (G^-1 by symmetric sweeps, entries of the
triangle on the block's threads) at the ranks where its layout changes: one
entry (M = 1), a few (M = 8, 36 entries in two warps), half the warps (M = 22),
every warp (M = 31, 496 entries) and more entries than threads (M = 32, 528), in
one uneven batch, against the oracle. Bounds as for the other fused tests: 1e-10
for FP64 and twice the FP32 random walk, 5e-5, for the FP32 state."""
import pytest

import lr_inputs as li
from oracle import parallel
from paper_2508_18114_gb300 import runner

from _compare import compare_observables

pytestmark = pytest.mark.gpu


def _filter(nt, nr, nf):
    import dataclasses
    return dataclasses.replace(li.c2().candidates[0].model, dims=(nt, nr, nf))


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32_g64", 5e-5)])
def test_ranks_at_the_edges_of_the_sweep(precision, tol):
    ranks = (1, 8, 22, 31, 32)
    cands = [li.Candidate(_filter(3 + k % 2, 6, 4), m, li.pulse_two_segment(60 + k, li.TWO_PI * 7.5))
             for k, m in enumerate(ranks)]
    wl = li.Workload("sweep_ranks", cands, 5e-4, 80, 0.4, init_seed=93, eps=1e-5)
    ora = parallel.run_workload(wl, None, 20)
    b = runner.make_batch(wl, precision=precision, engine="fused", pop_every=20)
    b.set_initial(wl.init_seed, wl.eps)
    b.integrate(wl.dt, wl.n_steps)
    got = b.observables()
    b.close()
    compare_observables(got, ora, 2 * len(ranks), [c.model.dims[0] for c in cands for _ in (0, 1)], tol, tol,
                        "sweep " + precision)
