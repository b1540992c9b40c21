"""Signal, photons, populations and trace that the FP32 sparse engine records, against
the FP64 contraction of the same FP32 state, in both schedules.

The readout operator has one entry per row, a power of two, so that r Z is exact
in FP32 and only the sums round. A thread or lane adds at most 48 exact products
and then 10 partial sums in double-word FP32 (2^-48 of the running sum each),
the rest is FP64: 64 x 2^-48 of the sum of the products' magnitudes.
"""
import numpy as np
import pytest

from paper_2508_18114_gb300.sparse import SparseBatch

pytestmark = pytest.mark.gpu

BOUND = 64 * 2.0 ** -48


def _model(N, n_levels):
    """A = 0 off the diagonal, one jump operator, r = one entry per row."""
    n = np.arange(N)
    col = np.concatenate([n, n, (7 * n + 3) % N])
    val = np.zeros((3 * N, 2))
    val[:N, 1] = -0.25
    val[N:2 * N, 0] = 0.5
    val[2 * N:, 0] = 2.0 ** ((n % 3) - 1)
    rowptr = np.concatenate([o * N + np.arange(N + 1) for o in range(3)])
    return dict(N=N, nnz=3 * N, n_jumps=1, n_levels=n_levels, wd=1.0, rowptr=rowptr, col=col, val=val.reshape(-1),
                chan=np.full(3 * N, 2), level=n % n_levels)


@pytest.mark.parametrize("wide", ["0", "1"])
@pytest.mark.parametrize("N,M,n_levels", [(33, 1, 2), (150, 20, 5), (640, 32, 16)])
def test_fp32_observables_are_summed_exactly(monkeypatch, N, M, n_levels, wide):
    monkeypatch.setenv("LR_SPARSE_WIDE", wide)
    model = _model(N, n_levels)
    T = 2
    b = SparseBatch(model, M, [(0, (1.0, 1.0, 0.01, 0.0))] * T, 0.05, 4, precision="fp32_g64")
    g = np.random.default_rng(11 * N + M)
    z = g.standard_normal((T, N, M)) + 1j * g.standard_normal((T, N, M))
    z = (z * 10.0 ** -np.linspace(0.0, 2.5, M)).astype(np.complex64).astype(np.complex128)
    b.set_state(z, 0)
    b.integrate(5e-4, 0)
    o = b.observables()
    y = z[:, (7 * np.arange(N) + 3) % N] * 2.0 ** ((np.arange(N) % 3) - 1)[None, :, None]
    size = (np.abs(z.real) + np.abs(z.imag)) * (np.abs(y.real) + np.abs(y.imag))
    row = (np.abs(z) ** 2).sum(2)
    for j in range(T):
        assert abs(o["beta"][j, 0] - (np.conj(z[j]) * y[j]).sum()) <= BOUND * size[j].sum()
        assert abs(o["nphot"][j, 0] - (np.abs(y[j]) ** 2).sum()) <= BOUND * (np.abs(y[j]) ** 2).sum()
        assert abs(o["trace"][j, 0] - row[j].sum()) <= BOUND * row[j].sum()
        want = np.array([row[j][model["level"] == k].sum() for k in range(n_levels)])
        assert np.abs(o["pops"][j, 0] - want).max() <= BOUND * row[j].sum()
