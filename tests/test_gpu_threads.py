"""Handles of one process on host threads of their own.  The kernels are shared
by all handles, and so is a kernel's limit on dynamic shared memory; two
handles whose sweeps ask for different amounts beyond the default 48 KB (FP64,
eight right-hand sides: 64 KB for the supernodes swept by a warp each, 70 KB for
those swept by a CTA with 480 rows below) solve at the same time, launch by
launch (profiling on: no graphs), on a stream each.  Nothing depends on timing:
the results are those of the same calls one after the other, bit for bit.
"""
import threading

import numpy as np
import pytest

from paper_2510_05885_gb300 import synth
from test_gpu_sweeps import _bordered, _lower, _t

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_two_handles_on_two_threads():
    from paper_2510_05885_gb300 import ncl_kkt as nk
    opts = dict(prec="fp64", subtree_sweeps=0, ir_max_iter=0, use_fgmres=0, ir_tol=1e-10)
    inst = synth.random_instance(20, 25, seed=31, form="stabilized", rho=1e4)
    p = inst.pat
    many = nk.KKT(0, p.n, p.m, p.H_rowptr, p.H_colind, p.J_rowptr, p.J_colind, **opts)
    many.factor(_t(inst.H_val), _t(inst.J_val), _t(inst.Sigma), inst.delta, inst.rho)
    A = _bordered(20, 12, 480, 5)
    n = len(A)
    ptr, col, val = _lower(A)
    z = np.zeros(1, np.int32)
    wide = nk.KKT(1, n, 0, ptr, col, z, z[:0], **opts)
    col0, _, nrow = wide.supernodes()
    assert any(c == 12 and r == 492 for c, r in zip(np.diff(col0), nrow))
    wide.factor(_t(val), None, _t(np.zeros(n)), 0.0, 1.0)
    jobs, bad = [], []
    for K in (many, wide, many, wide):
        if len(jobs) >= 2:      # the same two systems on handles of their own
            K = nk.KKT.like(K, **opts)
            args = (_t(inst.H_val), _t(inst.J_val), _t(inst.Sigma), inst.delta, inst.rho) if len(jobs) == 2 else \
                (_t(val), None, _t(np.zeros(n)), 0.0, 1.0)
            K.factor(*args)
        nk.ncl_kkt_profile(K._h, 1)
        B = _t(np.random.default_rng(7).standard_normal((K.dim, 8)))
        jobs.append((K, B, K.solve(B)[0].clone(), torch.cuda.Stream()))
    torch.cuda.synchronize()

    def work(K, B, want, stream):
        try:
            with torch.cuda.stream(stream):
                for _ in range(400):
                    if not torch.equal(K.solve(B)[0], want):
                        bad.append("another result")
                        return
        except Exception as e:   # noqa: BLE001 (reported below, on the test's own thread)
            bad.append(str(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    for K, *_ in jobs:
        K.close()
