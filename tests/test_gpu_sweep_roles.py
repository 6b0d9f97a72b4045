"""Sweep roles that depend on what else a level has: the same front alone (one
CTA up to 48 KB, strips beyond; a warp up to 512 entries below the pivots),
among 30 (several CTAs, each with a part of the rows below), among 153 (one CTA
whatever its size) and among 609 (a warp up to 4096 entries).  Every instance of a batch is solved without refinement; the bound is
the backward error of LDL^T factors in working precision, 8 n u for these
diagonally dominant matrices (3 n u times a growth below 2, rounded up).
"""
import numpy as np
import pytest

from test_gpu_sweeps import _bordered, _lower, _t

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32_ir", "fp64"])
@pytest.mark.parametrize("count,size,border", [(1, 120, 300), (30, 120, 300), (30, 128, 401), (153, 120, 300), (153, 100, 33), (1, 30, 100),
                                               (609, 30, 100), (609, 9, 40)])
def test_roles_by_level_size(count, size, border, prec):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    A = _bordered(1, size, border, 3)
    n = len(A)
    ptr, col, val = _lower(A)
    z = np.zeros(1, np.int32)
    K = nk.KKT.batch(1, [(n, 0, ptr, col, z, z[:0])] * count, prec=prec, subtree_sweeps=0, ir_max_iter=0,
                     use_fgmres=0, precision_fallback=0, ir_tol=1e-30)
    scale = 1.0 + np.arange(count) / count            # instance i is scale[i] A
    vals = _t((scale[:, None] * val[None]).reshape(-1))
    u = 2.0 ** -24 if prec == "fp32_ir" else 2.0 ** -53
    nrm = np.abs(A).sum(axis=1).max()
    for nrhs in (1, 3, 8):
        B = np.random.default_rng(nrhs).standard_normal((nrhs, count * n))
        X = torch.empty_like(_t(B))
        infos, _ = nk.ncl_kkt_batch_factor_solve(K._h, vals, None, _t(np.zeros(count * n)), [0.0] * count, [1.0] * count,
                                                 nrhs, _t(B), count * n, X, count * n)
        assert all(f.inertia == (n, 0, 0) for f in infos)
        X = X.cpu().numpy().reshape(nrhs, count, n) * scale[None, :, None]
        B = B.reshape(nrhs, count, n)
        R = np.abs(B - X @ A).max(axis=2)
        assert (R / (nrm * np.abs(X).max(axis=2) + np.abs(B).max(axis=2))).max() <= 8 * n * u
    K.close()
