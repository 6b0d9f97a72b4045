"""Factors whose multipliers are of order one and more, and pivots replaced by
the static pivot in the middle of coupled columns, on single dense fronts of
every kind.

The reference is the elimination without exchanges in numpy, with the same rule
for a tiny pivot: d with |d| <= eps becomes eps, and the factors are those of A +
E, E diagonal.  An unrefined solve is held to its own first-order bound, entry by
entry.  With u the unit roundoff, g = min(n, 4 sqrt(n)) u the error of a sum of n
products (the worst case for short ones, the probabilistic bound of Higham and
Mary, 2019, with lambda = 4 for long ones), M = L^-1 and y, z, x the exact forward,
diagonal and backward results:

  factors     g |L||D||L^T||x|
  inverse     the computed M is off by at most 2 g |M||L||M| (blocks of up to 128
              columns and their merges are each a product of at most n terms in
              either factor), a product with it adds g |M|: forward |L| (2 g
              |M||L||M| + g |M|) |b|, backward |L||D| times the same for |z|
  diagonal    u |L||D||z|

in all multiplied by 1.5 for what is of second order.  (FP32: quasi-definite
matrices of 65 columns and more are left out, where the bound says nothing.)
"""
import numpy as np
import pytest

from test_gpu_sweeps import _t

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [8, 20, 33, 64, 65, 129, 200, 257, 385]


def _eliminate(A, eps, vanish=()):
    """L, D of A + E, the number of replaced pivots; the pivots in `vanish` are
    made to vanish by changing A's own diagonal (in place)."""
    n = len(A)
    S, L, D, count = A.copy(), np.eye(n), np.zeros(n), 0
    for k in range(n):
        if k in vanish:
            A[k, k] -= S[k, k]
            S[k, k] = 0.0
        d = S[k, k]
        if abs(d) <= eps:
            assert abs(d) <= eps / 10
            d, count = eps, count + 1
        assert abs(d) >= 4 * eps or d == eps
        D[k] = d
        L[k + 1:, k] = S[k + 1:, k] / d
        S[k + 1:, k + 1:] -= np.outer(L[k + 1:, k], S[k, k + 1:])
    return L, D, count


def _bound(L, D, b, u):
    n = len(D)
    g = min(n, 4 * n ** 0.5) * u
    M = np.linalg.inv(L)
    z = (M @ b) / D
    x = M.T @ z
    aL, aM, aD = np.abs(L), np.abs(M), np.abs(D)
    inv = lambda v: 2 * g * (aM @ (aL @ (aM @ v))) + g * (aM @ v)            # noqa: E731
    inv_t = lambda v: 2 * g * (aM.T @ (aL.T @ (aM.T @ v))) + g * (aM.T @ v)  # noqa: E731
    mat = lambda v: aL @ (aD * (aL.T @ v))                                            # noqa: E731
    return 1.5 * (aL @ inv(np.abs(b)) + mat(inv_t(np.abs(z))) + u * (aL @ (aD * np.abs(z))) + g * mat(np.abs(x)))


def _matrix(kind, n, seed):
    """A in pivot order and the pivots that vanish."""
    rng = np.random.default_rng([seed, n])
    G = rng.standard_normal((n, n))
    if kind == "quasidefinite":
        m = n // 3
        H = G[m:, m:] @ G[m:, m:].T / n + np.eye(n - m)
        A = np.zeros((n, n))
        A[:n - m, :n - m] = H
        A[n - m:, :n - m] = G[:m, m:]
        A[:n - m, n - m:] = G[:m, m:].T
        A[n - m:, n - m:] = -1e-2 * np.eye(m)
        p = rng.permutation(n)
        return A[np.ix_(p, p)], ()
    if kind == "layered":      # three classes of columns, each coupled to the one before: M = I - N + N^2
        cls, L = rng.integers(0, 3, n), np.eye(n)
        for i in range(1, n):
            k = np.flatnonzero(cls[:i] == cls[i] - 1)
            k = rng.choice(k, min(3, len(k)), replace=False)
            L[i, k] = rng.choice([-1.0, 1.0], len(k)) * rng.uniform(0.5, 1.5, len(k))
        return (L * (rng.choice([-1.0, 1.0], n) * rng.uniform(1, 2, n))) @ L.T, ()
    A = 0.1 * min(1.0, (16 / n) ** 0.5) * np.tril(G, -1)   # against eps = 0.1: multipliers of order one below a replaced pivot
    A = A + A.T + np.diag(rng.uniform(6, 8, n))
    return A, tuple(sorted({min(3, n - 2), n // 2, n - 2}))


def _solve(A, prec, eps, sub, **kw):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    n = len(A)
    r, c = np.tril_indices(n)
    ptr = np.concatenate([[0], np.cumsum(np.arange(1, n + 1))]).astype(np.int32)
    z = np.zeros(1, np.int32)
    K = nk.KKT(1, n, 0, ptr, c.astype(np.int32), z, z[:0], prec=prec, subtree_sweeps=sub, pivot_eps=eps, ir_max_iter=0,
               use_fgmres=0, precision_fallback=0, ir_tol=1e-30, **kw)
    order = K.permutation
    P = np.empty_like(A)
    P[np.ix_(order, order)] = A
    info = K.factor(_t(P[r, c]), None, _t(np.zeros(n)), 0.0, 1.0)
    b = np.random.default_rng(n).standard_normal(n)
    pb = np.empty(n)
    pb[order] = b
    x = K.solve(_t(pb))[0].cpu().numpy()[order]
    K.close()
    return info, b, x


@pytest.mark.parametrize("prec", ["fp32_ir", "fp64"])
@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", ["quasidefinite", "layered", "vanishing"])
def test_unrefined_solve_within_its_bound(kind, n, prec):
    eps = 0.1 if kind == "vanishing" else 1e-10
    if kind == "quasidefinite" and prec == "fp32_ir" and n > 64:
        pytest.skip("the bound is above the right-hand side")
    A, vanish = _matrix(kind, n, 1)
    if prec == "fp32_ir":
        A = A.astype(np.float32).astype(np.float64)    # the values the factorisation sees
    L, D, count = _eliminate(A, eps, vanish)
    if prec == "fp32_ir":
        A = A.astype(np.float32).astype(np.float64)
        L, D, count = _eliminate(A, eps)
    assert count == len(vanish)
    E = np.diag((L * D) @ L.T - A)
    for sub in (0, 1):
        info, b, x = _solve(A, prec, eps, sub)
        assert info.inertia == (int((D > 0).sum()), int((D < 0).sum()), 0) and info.n_perturbed == count
        r = np.abs(b - A @ x - E * x)
        assert (r <= _bound(L, D, b, 2.0 ** -24 if prec == "fp32_ir" else 2.0 ** -53)).all(), (sub, r.max())


@pytest.mark.parametrize("prec", ["fp32_ir", "fp64"])
@pytest.mark.parametrize("sub", [0, 1])
@pytest.mark.parametrize("shape,front", [((12, 9, 40), (9, 49)), ((6, 30, 100), (30, 130)), ((4, 64, 90), (64, 154)),
                                         ((3, 96, 129), (96, 225)), ((3, 200, 30), (200, 230))], ids=str)
def test_replaced_pivots_above_rows_below(shape, front, sub, prec):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    leaves, size, border = shape
    n, eps = leaves * size + border, 0.1
    rng = np.random.default_rng([5, n])
    P = 0.1 * (16 / n) ** 0.5 * np.tril(rng.standard_normal((n, n)), -1)
    for k in range(leaves):
        P[(k + 1) * size:leaves * size, k * size:(k + 1) * size] = 0.0
    P = P + P.T + np.diag(rng.uniform(6, 8, n))
    r, c = np.nonzero(np.tril(P))
    ptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int32)
    z = np.zeros(1, np.int32)
    K = nk.KKT(1, n, 0, ptr, c.astype(np.int32), z, z[:0], prec=prec, subtree_sweeps=sub, pivot_eps=eps, ir_max_iter=0,
               use_fgmres=0, precision_fallback=0, ir_tol=1e-30)
    col0, _, nrow = K.supernodes()
    assert front in set(zip(np.diff(col0).tolist(), nrow.tolist()))
    order = K.permutation
    A = P[np.ix_(order, order)]
    vanish = (int(col0[0]) + size // 2, int(col0[1]), int(col0[-2]) + 1)
    cast = (lambda a: a.astype(np.float32).astype(np.float64)) if prec == "fp32_ir" else (lambda a: a)
    A = cast(A)
    _eliminate(A, eps, vanish)
    A = cast(A)
    L, D, count = _eliminate(A, eps)
    assert count == len(vanish)
    P[np.ix_(order, order)] = A
    info = K.factor(_t(P[r, c]), None, _t(np.zeros(n)), 0.0, 1.0)
    assert info.inertia == (int((D > 0).sum()), int((D < 0).sum()), 0) and info.n_perturbed == count
    b = rng.standard_normal(n)
    pb = np.empty(n)
    pb[order] = b
    x = K.solve(_t(pb))[0].cpu().numpy()[order]
    res = np.abs(b - A @ x - np.diag((L * D) @ L.T - A) * x)
    assert (res <= _bound(L, D, b, 2.0 ** -24 if prec == "fp32_ir" else 2.0 ** -53)).all(), res.max()
    K.close()
