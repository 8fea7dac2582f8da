"""The event's reductions where their blocks change: row and column marginals over 1, 8, 9,
64 and 65 parts (groups of 8 over 8 thread rows), entries around a block's 32, and more
samples than one pass of the marginals' last kernel covers.

Tolerances, before any run.  The stored ln Lbar and ln L^ML are FP32, and a tile sums its
pairs in FP32 with exponentials of ~2 ulp: a marginal differs from the FP64 sum of the stored
values by at most ~1e-6 relative plus FP32 roundings of ln Lbar, below 1e-4 in ln P for ln
Lbar up to 200.  The evidence's N_eff, N_eff,ext and N_eff,int against those from the
marginals (returned in FP32): 1e-3.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dpx():
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    ctx = dp.dotpe_create(0)
    yield dp, ctx
    dp.dotpe_destroy(ctx)


def _lse(a, axis=None):
    m = np.max(a, axis=axis, keepdims=True)
    s = np.log(np.sum(np.exp(a - m), axis=axis, keepdims=True)) + m
    return np.squeeze(s, axis=axis) if axis is not None else float(np.squeeze(s))


@pytest.mark.parametrize("rows,n_ext", [(1, 1), (127, 33), (129, 255), (1024, 257), (1153, 31), (8193, 65),
                                        (8300, 2049), (2, 33000)])
def test_marginals_sum_the_stored_values(dpx, rows, n_ext):
    dp, ctx = dpx
    wl = synth.make_workload(n_int=rows, n_ext=n_ext, n_det=2, n_modes=2, n_bins=33, snr=10.0, seed=rows % 97,
                             n_phi=4, ln_w="random")
    bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m, wl.bank.ln_w)
    try:
        eid = dp.dotpe_event_submit(ctx, bid, 0, rows, wl.event.psd, wl.event.data, wl.ext.t, wl.ext.R, wl.ext.ln_w,
                                    n_phi=4, u_min=wl.event.u_min, precision="fp16x3",
                                    flags=dp.DOTPE_FLAG_STORE_LNL)
        dp.dotpe_event_wait(ctx, eid, 60.0)
        ev = dp.dotpe_evidence(ctx, eid)
        lnl, row, col = (dp.dotpe_lnl_blocks(ctx, eid, 0, rows, 0, n_ext, what=w)
                         for w in (dp.DOTPE_LNL_MARG, dp.DOTPE_ROW_MARGINAL, dp.DOTPE_COL_MARGINAL))
        dp.dotpe_event_release(ctx, eid)
    finally:
        dp.dotpe_bank_release(ctx, bid)
    assert np.max(np.abs(lnl)) < 200.0
    lp = lnl.astype(np.float64) + wl.bank.ln_w[:, None] + wl.ext.ln_w[None, :] + np.log(4.0)
    assert np.max(np.abs(row - _lse(lp, 1))) <= 1e-4
    assert np.max(np.abs(col - _lse(lp, 0))) <= 1e-4
    row, col = row.astype(np.float64), col.astype(np.float64)
    s1 = _lse(lp)
    assert abs(ev["ln_z"] - (s1 - np.log(rows) - np.log(n_ext) - np.log(4))) <= 1e-4
    assert ev["n_eff_int"] == pytest.approx(np.exp(2 * s1 - _lse(2 * row)), rel=1e-3)
    assert ev["n_eff_ext"] == pytest.approx(np.exp(2 * s1 - _lse(2 * col)), rel=1e-3)
