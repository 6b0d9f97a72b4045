"""FP32 pivots near the ends of the exponent range, with nonzero multipliers: A =
L D L^T, L with 1/2 and 1/4 below the diagonal at distances 1 and 9 (within a
panel of eight columns and across), D powers of two between 2^125 and 2^127, or
2^-127 and 2^-125.  Every entry of A, L and D has a few bits, so the factors are
exact where the elimination is right; an unrefined solve is held to 8 n u as in
test_gpu_sweeps.  A reciprocal that loses the pivot 2^127 drops whole
multipliers: an error of order one.
"""
import numpy as np
import pytest

from test_gpu_sweeps import _t

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sub", [0, 1])
@pytest.mark.parametrize("n", [7, 16, 30, 60, 150, 200])
@pytest.mark.parametrize("exps,scale", [((125, 127, 126), 2.0 ** -4), ((-125, -127, -126), 16.0)], ids=["large", "small"])
def test_extreme_pivots(exps, scale, n, sub):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    d = 2.0 ** np.resize(np.array(exps, dtype=float), n)
    L = np.eye(n) + 0.5 * np.eye(n, k=-1) + 0.25 * np.eye(n, k=-9)
    A = (L * d) @ L.T
    r, c = np.tril_indices(n)                       # one dense front
    ptr = np.concatenate([[0], np.cumsum(np.arange(1, n + 1))]).astype(np.int32)
    z = np.zeros(1, np.int32)
    K = nk.KKT(1, n, 0, ptr, c.astype(np.int32), z, z[:0], prec="fp32_ir", subtree_sweeps=sub, pivot_eps=1e-44,
               ir_max_iter=0, use_fgmres=0, precision_fallback=0, ir_tol=1e-30)
    order = K.permutation                           # pivot k is row order[k]: permute so that L stays as it is
    P = np.empty_like(A)
    P[np.ix_(order, order)] = A
    info = K.factor(_t(P[r, c]), None, _t(np.zeros(n)), 0.0, 1.0)
    assert info.inertia == (n, 0, 0) and info.n_perturbed == 0
    b = P @ np.where(np.arange(n) % 3, scale, -scale)
    x = K.solve(_t(b))[0].cpu().numpy()
    eta = np.abs(b - P @ x).max() / (np.abs(P).sum(axis=1).max() * np.abs(x).max() + np.abs(b).max())
    assert eta <= 8 * n * 2.0 ** -24
    K.close()
