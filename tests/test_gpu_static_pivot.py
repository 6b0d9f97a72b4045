"""Static pivoting inside the pivot blocks, at the edges of the eight-column
panels: an exactly zero pivot at a chosen column of a diagonal matrix (the
elimination leaves the others untouched) in fronts of every kind, perturbed
or reported under the stop policy, with the other pivots and the solution
unaffected; and a non-finite value refused.

The matrix is diag(d) with one dense coupling that makes it a single front:
A = D + B with B zero, entered as an explicit pattern of zeros, so the
factorisation is exact and every expected number is known beforehand.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda:0")


def _handle(n, prec, **kw):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    r, c = np.tril_indices(n)
    ptr = np.concatenate([[0], np.cumsum(np.arange(1, n + 1))]).astype(np.int32)
    z = np.zeros(1, np.int32)
    return nk.KKT(1, n, 0, ptr, c.astype(np.int32), z, z[:0], prec=prec, precision_fallback=0, **kw), r, c


@pytest.mark.parametrize("prec", ["fp32_ir", "fp64"])
@pytest.mark.parametrize("n", [5, 8, 20, 33, 64, 65, 120, 129, 150])
def test_zero_pivot_is_perturbed_or_reported(n, prec):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    for sub in (0, 1):
        K, r, c = _handle(n, prec, subtree_sweeps=sub, ir_max_iter=0, use_fgmres=0)
        stop, _, _ = _handle(n, prec, subtree_sweeps=sub, pivot_policy=nk.PIVOT_STOP)
        d = 1.0 + np.arange(n) % 4
        for at in sorted({0, 3, 7 % n, 8 % n, n // 2, n - 1}):
            v = np.zeros(len(r))
            diag = d.copy()
            diag[at] = 0.0
            v[r == c] = diag
            info = K.factor(_t(v), None, _t(np.zeros(n)), 0.0, 1.0)
            assert info.inertia == (n, 0, 0) and info.n_perturbed == 1
            b = np.ones(n)
            b[at] = 0.0     # consistent with the zero row
            X, _ = K.solve(_t(b))
            want = np.where(diag > 0, 1.0 / np.where(diag > 0, diag, 1.0), 0.0)
            # powers of two and a third: one division's rounding
            assert np.abs(X.cpu().numpy() - want).max() <= (2.0 ** -24 if prec == "fp32_ir" else 2.0 ** -53)
            fs = stop.factor(_t(v), None, _t(np.zeros(n)), 0.0, 1.0)
            assert fs.status == nk.ERR_ZERO_PIVOT and fs.inertia == (n - 1, 0, 1)
            diag[at] = -2.0
            v[r == c] = diag
            assert K.factor(_t(v), None, _t(np.zeros(n)), 0.0, 1.0).inertia == (n - 1, 1, 0)
        v[r == c] = np.where(np.arange(n) == n // 2, np.inf, d)
        with pytest.raises(nk.NclError) as e:
            K.factor(_t(v), None, _t(np.zeros(n)), 0.0, 1.0)
        assert e.value.status == 7
        K.close()
        stop.close()
