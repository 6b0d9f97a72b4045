"""Front assembly at the edge of what shared memory holds: an FP64 front of
4109 rows, whose rows up to 4096 entries are put together there (one to a CTA)
and longer ones in global memory, with a child under it; and fronts of a few
rows with several children.  Unrefined solves, 8 n u as in test_gpu_sweeps.
"""
import numpy as np
import pytest

from test_gpu_sweeps import _bordered, _lower, _t

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,leaves,size,border", [("fp64", 1, 8, 4101), ("fp32_ir", 1, 8, 1200), ("fp64", 5, 3, 31),
                                                     ("fp32_ir", 5, 3, 33), ("fp32_ir", 2, 5, 64)])
def test_assembly(prec, leaves, size, border):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    A = _bordered(leaves, size, border, 9)
    n = len(A)
    ptr, col, val = _lower(A)
    z = np.zeros(1, np.int32)
    K = nk.KKT(1, n, 0, ptr, col, z, z[:0], prec=prec, subtree_sweeps=0, ir_max_iter=0, use_fgmres=0,
               precision_fallback=0, ir_tol=1e-30)
    u = 2.0 ** -24 if prec == "fp32_ir" else 2.0 ** -53
    for scale in (1.0, 3.0):      # the second call meets the first one's fronts
        info = K.factor(_t(scale * val), None, _t(np.zeros(n)), 0.0, 1.0)
        assert info.inertia == (n, 0, 0)
        b = np.random.default_rng(2).standard_normal(n)
        x = K.solve(_t(b))[0].cpu().numpy() * scale
        eta = np.abs(b - A @ x).max() / (np.abs(A).sum(axis=1).max() * np.abs(x).max() + np.abs(b).max())
        assert eta <= 8 * n * u
    K.close()
