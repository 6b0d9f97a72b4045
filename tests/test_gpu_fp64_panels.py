"""FP64 fronts at the edges of their 32-column panels and 32-row tiles, and
pivots near the ends of the exponent range.

Unrefined solves are held to the normwise backward error of LDL^T factors in
double precision, 8 n u for these diagonally dominant matrices (n the order,
u = 2^-53: 3 n u times a growth below 2, rounded up).  A diagonal matrix loses
one rounding to the reciprocal and one to the product: 2 u, 3 u asked.
"""
import numpy as np
import pytest

from test_gpu_sweeps import _bordered, _dense, _lower, _t

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("persistent", [0, 1])
@pytest.mark.parametrize("case", [(1, 70, 1), (1, 95, 33), (2, 96, 31), (2, 97, 64), (1, 65, 129), (2, 63, 32), (3, 31, 8),
                                  (2, 33, 7), (1, 40, 200), (0, 300, 0)], ids=str)
def test_panels(case, persistent):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    leaves, size, border = case
    A = _bordered(leaves, size, border, 11) if leaves else _dense(size, 11)
    n = len(A)
    ptr, col, val = _lower(A)
    z = np.zeros(1, np.int32)
    K = nk.KKT(1, n, 0, ptr, col, z, z[:0], prec="fp64", persistent_fronts=persistent, ir_max_iter=0, use_fgmres=0)
    info = K.factor(_t(val), None, _t(np.zeros(n)), 0.0, 1.0)
    assert info.inertia == (n, 0, 0)
    b = np.random.default_rng(5).standard_normal(n)
    x = K.solve(_t(b))[0].cpu().numpy()
    eta = np.abs(b - A @ x).max() / (np.abs(A).sum(axis=1).max() * np.abs(x).max() + np.abs(b).max())
    assert eta <= 8 * n * 2.0 ** -53
    K.close()


def test_extreme_pivots():
    from paper_2510_05885_gb300 import ncl_kkt as nk
    n = 72
    r, c = np.tril_indices(n)
    ptr = np.concatenate([[0], np.cumsum(np.arange(1, n + 1))]).astype(np.int32)
    z = np.zeros(1, np.int32)
    K = nk.KKT(1, n, 0, ptr, c.astype(np.int32), z, z[:0], prec="fp64", pivot_eps=1e-305, ir_max_iter=0, use_fgmres=0)
    e = np.resize([-303, -291, -289, -200, -12, 0, 9, 200, 289, 291, 305], n)
    d = (1.0 + np.arange(n) / 97.0) * 10.0 ** e * np.where(np.arange(n) % 3, 1.0, -1.0)
    v = np.zeros(len(r))
    v[r == c] = d
    info = K.factor(_t(v), None, _t(np.zeros(n)), 0.0, 1.0)
    assert info.inertia == (int((d > 0).sum()), int((d < 0).sum()), 0) and info.n_perturbed == 0
    for scale in (1.0, 1e-9):
        b = np.full(n, scale) * d      # subnormal entries have lost bits: compare with b as it is
        x = K.solve(_t(b))[0].cpu().numpy()
        assert np.abs(x / (b / d) - 1.0).max() <= 3 * 2.0 ** -53
    K.close()
