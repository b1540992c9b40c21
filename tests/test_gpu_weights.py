"""The couplings of the whole-chip kernels on an FP32 state are rounded once.

Column m of the state is one basis state |n_m>. One step of size h = 2^-30 takes it
to -i h H_kn |n_m> in the rows k that g or J couples it to (second-order terms are
below 2^-50 of that), through RK4 sums of w, w + 2w, .. and a product with h / 6 whose
roundings are known. So the entry tells w to the last bit: it has to be the FP32 number
next to the coupling, g sqrt(i j), that FP64 gives.
"""
import numpy as np
import pytest

import lr_inputs as li
from paper_2508_18114_gb300 import runner

pytestmark = pytest.mark.gpu

H = 2.0 ** -30
f32 = np.float32


def _step(w):
    """FP32 image of an RK4 step of dz/dt = w from 0 (each fma rounds an exact product)."""
    fma = lambda a, b, c: f32(float(a) * float(b) + float(c))  # noqa: E731  (exact in FP64 up to 2^-53)
    s = fma(2, w, w)
    s = fma(2, w, s)
    s = fma(1, w, s)
    hi = f32(H / 6)
    return fma(f32(H / 6 - float(hi)), s, f32(float(hi) * float(s)))


@pytest.mark.parametrize("dims,frame", [((6, 9, 5), "lab"), ((6, 9, 5), "rwa"), ((5, 60), "lab")])
def test_couplings_of_an_fp32_state_round_once(monkeypatch, dims, frame):
    gc, J = 0.9437, 0.6291
    m = li.ModelParams(dims=dims, wq=0.2, alpha=-0.1, wr=0.3, g=gc, kappa=0.01, gamma=1e-3,
                       **({"wf": 0.25, "J": J} if len(dims) == 3 else {}))
    M = 12
    wl = li.Workload("weights", [li.Candidate(m, M, li.PulseParams(0, (0.0, 0.3, 0.01, 0.0)))], H, 1, 1.0,
                     init_seed=1, eps=1e-4, frame=frame)
    N = int(np.prod(dims))
    rows = np.random.default_rng(3).permutation(N)[:M]
    z = np.zeros((N, M), complex)
    z[rows, np.arange(M)] = 1.0
    monkeypatch.setenv("LR_FUSED_WIDE", "1")
    b = runner.make_batch(wl, precision="fp32_g64", engine="fused", pop_every=1, max_steps=1)
    for j in (0, 1):
        b.set_state(j, z, 0)
    b.integrate(H, 1)
    out = b.get_state(0)
    b.close()
    full = dims if len(dims) == 3 else (*dims, 1)
    seen = 0
    for mcol, n in enumerate(rows):
        it, ir, i_f = np.unravel_index(n, full)
        for a in (-1, 1):
            for c in (-1, 1):
                if frame == "rwa" and a == c:
                    continue
                for k, w in (((it + a, ir + c, i_f), gc * np.sqrt(max(it, it + a)) * np.sqrt(max(ir, ir + c))),
                             ((it, ir + a, i_f + c), J * np.sqrt(max(ir, ir + a)) * np.sqrt(max(i_f, i_f + c)))):
                    if min(k) < 0 or any(x >= y for x, y in zip(k, full)):
                        continue
                    got = out[np.ravel_multi_index(k, full), mcol].imag
                    assert got == -float(_step(f32(w))), (n, k, w)
                    seen += 1
    assert seen >= 30
