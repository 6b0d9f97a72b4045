"""Leaves of small subtrees, which a warp factors where they fit its share of
the shared memory and a CTA otherwise: leaves of 1 to 32 pivots with up to 90
rows below, all coupled to one border.  Unrefined solves, 8 n u as in
test_gpu_sweeps; an exactly zero pivot in a leaf is perturbed and counted.
"""
import numpy as np
import pytest

from test_gpu_sweeps import _dominant, _lower, _t

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _leaves(sizes, border, seed):
    rng = np.random.default_rng(seed)
    n = sum(sizes) + border
    A = np.zeros((n, n))
    at = 0
    for k in sizes:
        A[at:at + k, at:at + k] = np.tril(rng.standard_normal((k, k)), -1)
        at += k
    A[at:, :at] = rng.standard_normal((border, at))
    A[at:, at:] = np.tril(rng.standard_normal((border, border)), -1)
    return _dominant(A)


@pytest.mark.parametrize("prec", ["fp32_ir", "fp64"])
@pytest.mark.parametrize("sizes,border", [((1, 2, 3, 4, 5, 6, 7, 8), 34), ((6, 6, 6, 12, 17, 18), 62), ((9, 24, 31, 32), 90),
                                          ((5,) * 40, 35), ((8, 16, 8), 33)])
def test_leaves(sizes, border, prec):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    A = _leaves(sizes, border, 4)
    n = len(A)
    ptr, col, val = _lower(A)
    z = np.zeros(1, np.int32)
    K = nk.KKT(1, n, 0, ptr, col, z, z[:0], prec=prec, subtree_sweeps=1, ir_max_iter=0, use_fgmres=0,
               precision_fallback=0, ir_tol=1e-30)
    u = 2.0 ** -24 if prec == "fp32_ir" else 2.0 ** -53
    for scale in (1.0, 3.0):
        info = K.factor(_t(scale * val), None, _t(np.zeros(n)), 0.0, 1.0)
        assert info.inertia == (n, 0, 0)
        b = np.random.default_rng(2).standard_normal(n)
        x = K.solve(_t(b))[0].cpu().numpy() * scale
        eta = np.abs(b - A @ x).max() / (np.abs(A).sum(axis=1).max() * np.abs(x).max() + np.abs(b).max())
        assert eta <= 8 * n * u
    # zero values but for the diagonal: the elimination leaves every pivot as it is
    r = np.repeat(np.arange(n), np.diff(ptr))
    d = 1.0 + np.arange(n) % 4
    for at in (0, sizes[0], sum(sizes) - 1):
        e = d.copy()
        e[at] = 0.0
        v = np.where(r == col, e[r], 0.0)
        info = K.factor(_t(v), None, _t(np.zeros(n)), 0.0, 1.0)
        assert info.inertia == (n, 0, 0) and info.n_perturbed == 1
    K.close()
