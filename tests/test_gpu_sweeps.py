"""Triangular sweeps and pivot-block inverses at the edges of their roles and
tiles, through the C ABI: single dense fronts around the 32-, 64-, 128- and
256-column boundaries, bordered systems whose border pulls updates from many
children, and every compiled number of right-hand sides.

The bound on an unrefined solve is the normwise backward error of LDL^T
factors applied in working precision, 3 n u (n the order, u = 2^-24 or 2^-53)
times the growth |L||D||L^T| / |A|, at most n for these diagonally dominant
matrices but in fact below 2; 8 n u is asked.  A refinement step then gains at
least 1 / (8 n u kappa) with kappa < 10, so two steps reach 1e-10 (n <= 400:
8 n u kappa < 2e-3 in FP32) and none is needed for 1e-12 in FP64.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda:0")


def _lower(A):
    n = A.shape[0]
    mask = np.tril(A != 0)
    ptr = np.concatenate([[0], np.cumsum(mask.sum(axis=1))]).astype(np.int32)
    r, c = np.nonzero(mask)
    return ptr, c.astype(np.int32), A[r, c]


def _dominant(A):
    A = A + A.T
    A[np.arange(len(A)), np.arange(len(A))] = 1.5 * np.abs(A).sum(axis=1) + 1.0
    return A


def _dense(n, seed):
    return _dominant(np.tril(np.random.default_rng(seed).standard_normal((n, n)), -1))


def _bordered(leaves, size, border, seed):
    """`leaves` dense blocks of `size`, each coupled to the whole border."""
    rng = np.random.default_rng(seed)
    n = leaves * size + border
    A = np.zeros((n, n))
    for k in range(leaves):
        s = slice(k * size, (k + 1) * size)
        A[s, s] = np.tril(rng.standard_normal((size, size)), -1)
    A[leaves * size:, :leaves * size] = rng.standard_normal((border, leaves * size))
    A[leaves * size:, leaves * size:] = np.tril(rng.standard_normal((border, border)), -1)
    return _dominant(A)


CASES = [("dense", n) for n in (1, 2, 4, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128, 129, 160, 255, 256, 257, 385)] + \
        [("bordered", 3, 5, 4), ("bordered", 9, 20, 33), ("bordered", 4, 40, 130), ("bordered", 3, 70, 70)]


@pytest.mark.parametrize("prec", ["fp32_ir", "fp64"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_sweeps_at_role_and_tile_edges(case, prec):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    A = _dense(case[1], case[1]) if case[0] == "dense" else _bordered(*case[1:], seed=case[1])
    n = len(A)
    ptr, idx, val = _lower(A)
    z = np.zeros(1, np.int32)
    u = 2.0 ** -24 if prec == "fp32_ir" else 2.0 ** -53
    nrm = np.abs(A).sum(axis=1).max()
    rng = np.random.default_rng(5)
    for sub in (0, 1):
        raw = nk.KKT(1, n, 0, ptr, idx, z, z[:0], prec=prec, subtree_sweeps=sub, ir_max_iter=0, use_fgmres=0,
                     precision_fallback=0, ir_tol=1e-30)
        ref = nk.KKT(1, n, 0, ptr, idx, z, z[:0], prec=prec, subtree_sweeps=sub)
        for K in (raw, ref):
            info = K.factor(_t(val), None, _t(np.zeros(n)), 0.0, 1.0)
            assert info.inertia == (n, 0, 0)
        for nrhs in (1, 2, 3, 4, 5, 8, 9):
            B = rng.standard_normal((n, nrhs))
            X, _ = raw.solve(_t(B))
            X = X.cpu().numpy()
            for r in range(nrhs):
                eta = np.abs(B[:, r] - A @ X[:, r]).max() / (nrm * np.abs(X[:, r]).max() + np.abs(B[:, r]).max())
                assert eta <= 8 * n * u, (sub, nrhs, r, eta)
            X, si = ref.solve(_t(B))
            assert si.status == 0 and si.used_fgmres == 0
            assert si.ir_iters <= (2 if prec == "fp32_ir" else 0)
        raw.close()
        ref.close()
