"""Event preparation at the edges of its blocks: one to nine samples around the blocks of
four (mode banks) and two (polarisations), odd and even numbers of bins around the lanes'
pairs of columns and the blocks of 128 bins, one to four modes, the FP32, one- and two-plane
operands; and with relative-binning weights of a polarisation-resolved bank.

Tolerance, before any run: the split and FP32 precisions' |d ln Lbar|, |d ln L^ML| <= 1e-3
per pair against the oracle.
"""
import numpy as np
import pytest

import oracle
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


def _check(dp, ctx, wl, precision, rb=None, F=None):
    I, E = wl.bank.h.shape[0], wl.ext.t.shape[0]
    ref, _ = oracle.OracleProblem(wl.bank, wl.ext, wl.event, rb=rb).eval_grid(0.0)
    bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m, wl.bank.ln_w)
    try:
        psd, data = (wl.event.psd, wl.event.data) if rb is None else (None, None)
        eid = dp.dotpe_event_submit(ctx, bid, 0, I, psd, data, wl.ext.t, None if F is not None else wl.ext.R,
                                    wl.ext.ln_w, n_phi=wl.event.n_phi, u_min=wl.event.u_min, precision=precision,
                                    flags=dp.DOTPE_FLAG_STORE_LNL, rb=rb, F=F)
        dp.dotpe_event_wait(ctx, eid, 60.0)
        lnl, ml = (dp.dotpe_lnl_blocks(ctx, eid, 0, I, 0, E, w) for w in (dp.DOTPE_LNL_MARG, dp.DOTPE_LNL_ML_MAX))
        dp.dotpe_event_release(ctx, eid)
    finally:
        dp.dotpe_bank_release(ctx, bid)
    assert np.max(np.abs(lnl - ref["lnl_marg"])) <= 1e-3
    assert np.max(np.abs(ml - ref["lnl_ml_max"])) <= 1e-3


@pytest.mark.parametrize("precision", ["fp32", "bf16x3", "fp16x3"])
@pytest.mark.parametrize("n_ext,bins,modes,n_det", [
    (1, 31, 1, 1), (2, 32, 2, 2), (3, 33, 3, 3), (4, 64, 4, 2), (5, 127, 4, 3), (7, 128, 2, 1), (8, 129, 3, 2),
    (9, 255, 4, 3), (33, 257, 1, 2)])
def test_mode_banks(dpx, n_ext, bins, modes, n_det, precision):
    dp, ctx = dpx
    wl = synth.make_workload(n_int=3, n_ext=n_ext, n_det=n_det, n_modes=modes, n_bins=bins, snr=12.0,
                             seed=bins + n_ext, ln_w="random")
    _check(dp, ctx, wl, precision)


@pytest.mark.parametrize("precision", ["bf16x3", "fp16x3"])
@pytest.mark.parametrize("n_ext,bins,modes,n_det", [(1, 33, 1, 1), (3, 64, 2, 3), (4, 97, 4, 2), (5, 129, 3, 3)])
def test_polarisations_with_weights(dpx, n_ext, bins, modes, n_det, precision):
    dp, ctx = dpx
    rw = synth.make_rb_workload(3, n_ext, n_det, modes, bins, n_fine=16384, snr=12.0, seed=bins, precessing=True)
    w = oracle.rb_weights(rw.f_fine, rw.dff, rw.psd_fine, rw.data_fine, rw.h0_fine, rw.nodes, rw.t0)
    _check(dp, ctx, rw, precision, rb=w, F=rw.ext.F)
