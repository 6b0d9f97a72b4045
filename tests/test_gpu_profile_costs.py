"""The profile's operations of the pivot blocks' inverses: w^3 / 3 for a dense
front of w columns up to 128, and for wider ones the sum over its 128-column
blocks (FP32: the merges of the blocks apart).
"""
import numpy as np
import pytest

from test_gpu_sweeps import _dense, _lower, _t

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32_ir", "fp64"])
@pytest.mark.parametrize("n", [40, 100, 300])
def test_inverse_costs(n, prec):
    from paper_2510_05885_gb300 import ncl_kkt as nk
    A = _dense(n, n)
    ptr, col, val = _lower(A)
    z = np.zeros(1, np.int32)
    K = nk.KKT(1, n, 0, ptr, col, z, z[:0], prec=prec, subtree_sweeps=0)
    nk.ncl_kkt_profile(K._h, 1)
    K.factor(_t(val), None, _t(np.zeros(n)), 0.0, 1.0)
    rep = nk.ncl_kkt_profile_report(K._h)
    inv = rep["invert_blocks_f32" if prec == "fp32_ir" else "invert_blocks_f64"]
    w = np.array([min(128, n - b) for b in range(0, n, 128)], dtype=float)
    assert inv["launches"] == 1
    assert inv["flops"] == pytest.approx((w ** 3).sum() / 3, rel=1e-6)
    assert inv["bytes"] == pytest.approx((w * w).sum() * (4 if prec == "fp32_ir" else 8), rel=1e-6)
    assert (rep.get("invert_merge_f32", {"flops": 0})["flops"] > 0) == (prec == "fp32_ir" and n > 128)
    K.close()
