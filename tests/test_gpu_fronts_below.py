"""Fronts with rows below their pivots, in every role of the panels, the inverses
and the sweeps.  Blocks coupled to one border merge into a single front where
they are few (relaxed amalgamation), so each case states the front it is meant
to have and is refused without it:

  roles    the same front where a level has little work (a warp up to 512
           entries below, a CTA up to 48 KB, strips beyond) and in a batch with
           more (a CTA for any front, forward several with a part of the rows
           each; a warp up to 4096 entries)
  panels   row CTAs of 32 and 64 rows at their edges
  chunks   staged vectors longer than a chunk of 64 KB (eight right-hand sides:
           2048 entries in FP32, 1024 in FP64): pivot rows, rows below and both
           column sums; pivot blocks of more than 1024 columns, whose inverses
           merge from blocks of 128 to 2048
  merges   more merge items in one launch than are done in the finer tiles
  assembly children under a front whose rows are put together one to a CTA and,
           above 4096 entries (FP64), in global memory

Unrefined solves are held to 8 n u as in test_gpu_sweeps (u = 2^-24 or 2^-53).
"""
import numpy as np
import pytest

from test_gpu_sweeps import _bordered, _dense, _lower, _t

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(A, count, prec, nrhs, front=None, **opts):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    n = len(A)
    ptr, col, val = _lower(A)
    z = np.zeros(1, np.int32)
    K = nk.KKT.batch(1, [(n, 0, ptr, col, z, z[:0])] * count, prec=prec, ir_max_iter=0, use_fgmres=0,
                     precision_fallback=0, ir_tol=1e-30, **opts)
    if front:
        col0, _, nrow = K.supernodes()
        assert front in set(zip(np.diff(col0).tolist(), nrow.tolist()))
    scale = 1.0 + np.arange(count) / count            # instance i is scale[i] A
    vals = _t((scale[:, None] * val[None]).reshape(-1))
    u = 2.0 ** -24 if prec == "fp32_ir" else 2.0 ** -53
    nrm = np.abs(A).sum(axis=1).max()
    for nr in nrhs:
        B = np.random.default_rng(nr).standard_normal((nr, count * n))
        X = torch.empty_like(_t(B))
        infos, _ = nk.ncl_kkt_batch_factor_solve(K._h, vals, None, _t(np.zeros(count * n)), [0.0] * count, [1.0] * count,
                                                 nr, _t(B), count * n, X, count * n)
        assert all(f.inertia == (n, 0, 0) for f in infos)
        X = X.cpu().numpy().reshape(nr, count, n) * scale[None, :, None]
        B = B.reshape(nr, count, n)
        R = np.abs(B - X @ A).max(axis=2)
        assert (R / (nrm * np.abs(X).max(axis=2) + np.abs(B).max(axis=2))).max() <= 8 * n * u
    K.close()


@pytest.mark.parametrize("prec", ["fp32_ir", "fp64"])
@pytest.mark.parametrize("count,shape,front", [(1, (12, 9, 40), (9, 49)), (1, (20, 12, 480), (12, 492)),
                                               (1, (6, 30, 100), (30, 130)), (130, (6, 30, 100), (30, 130)),
                                               (1, (6, 100, 300), (100, 400)), (30, (6, 100, 300), (100, 400)),
                                               (1, (4, 128, 401), (128, 529)), (8, (4, 128, 401), (128, 529)),
                                               (4, (3, 200, 30), (200, 230))], ids=str)
def test_roles(count, shape, front, prec):
    _check(_bordered(*shape, seed=3), count, prec, (1, 3, 8), front, subtree_sweeps=0)


@pytest.mark.parametrize("persistent", [0, 1])
@pytest.mark.parametrize("prec", ["fp32_ir", "fp64"])
@pytest.mark.parametrize("shape,front", [((4, 60, 500), (60, 560)), ((6, 40, 300), (40, 340)), ((4, 64, 90), (64, 154)),
                                         ((3, 96, 129), (96, 225)), ((3, 97, 64), (97, 161)), ((4, 300, 1100), (300, 1400))],
                         ids=str)
def test_panels(shape, front, prec, persistent):
    _check(_bordered(*shape, seed=4), 1, prec, (1,), front, persistent_fronts=persistent)


@pytest.mark.parametrize("prec,shape,front", [("fp32_ir", (2, 2100, 40), (2100, 2140)), ("fp32_ir", (2, 600, 2100), (600, 2700)),
                                              ("fp64", (2, 1100, 300), (1100, 1400)), ("fp64", (4, 300, 1100), (300, 1400))],
                         ids=str)
def test_chunks(prec, shape, front):
    _check(_bordered(*shape, seed=5), 1, prec, (1, 5, 8), front)


@pytest.mark.parametrize("n", [129, 200])
def test_many_merges(n):
    _check(_dense(n, n), 320, "fp32_ir", (1,))


def test_assembly_of_long_rows():
    _check(_bordered(2, 600, 3550, seed=6), 1, "fp64", (1,), (600, 4150))
