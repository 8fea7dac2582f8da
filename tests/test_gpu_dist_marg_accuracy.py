"""The distance marginal against the FP64 oracle where its table interpolates worst: small s,
y where the peak sets in.

The interpolation error is the same for neighbouring arguments, the FP32 roundings differ:
averages over small boxes of (y, ln s) show the former.  Tolerance, before any run: the node
table's bicubic is within 6.1e-6 of 64-bit quadrature for ln s in [-6, -4] and the cells are
restrictions of it; their coefficients are FP32 (below 32: 1e-6 each way); 200 roundings of
3e-6 rms average to 2.1e-7, five sigma 1.1e-6.  Together 8.2e-6.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def test_boxes_where_the_peak_sets_in():
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    u_min = float(np.float32(0.37))
    rng = np.random.default_rng(3)
    ny, ns, per = 160, 8, 200  # boxes of 1/64 x 1/16
    y = 4.5 + (np.arange(ny)[:, None, None] + rng.random((ny, ns, per))) / 64
    sig = -6.0 + (np.arange(ns)[None, :, None] + rng.random((ny, ns, per))) / 16
    s = np.exp(sig)
    hh = ((s / u_min) ** 2).astype(np.float32)
    dh = ((y + s) * s / u_min).astype(np.float32)
    ctx = dp.dotpe_create(0)
    try:
        got = dp.dotpe_dist_marg_eval(ctx, dh.ravel(), hh.ravel(), u_min).astype(np.float64)
    finally:
        dp.dotpe_destroy(ctx)
    ref = np.array([oracle.dist_marg(float(a), float(b), u_min) for a, b in zip(dh.ravel(), hh.ravel())])
    off = (got - ref).reshape(ny, ns, per).mean(axis=2)
    print("largest mean error of a box %.3g" % np.max(np.abs(off)))
    assert np.max(np.abs(off)) <= 8.2e-6
