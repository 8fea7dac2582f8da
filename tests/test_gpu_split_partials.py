"""Split-precision events (separate low-order accumulator): the row, column and total sums
hold every pair of every tile.

A tile's epilogue warps take interleaved samples of the tile's two 16-sample halves and
collect their pairs' values in one shared array; an entry lost there leaves the stored pair
as it is and falls out of the sums.  Few bins and modes keep the tensor-core part short, so
the warps are as far apart as they get; many tiles per SM; a quiet event, so that every pair
has a share in its row and column.

Tolerance, before any run: stored ln Lbar are FP32 and below 50 here (roundings of 4e-6), a
tile's FP32 sums carry ~1e-6 and the returned marginals are FP32: 5e-5 in ln P.  A pair lost
from a row of 161 or a column of 5,000 moves it by its share.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _lse(a, axis=None):
    m = np.max(a, axis=axis, keepdims=True)
    s = np.log(np.sum(np.exp(a - m), axis=axis, keepdims=True)) + m
    return np.squeeze(s, axis=axis) if axis is not None else float(np.squeeze(s))


@pytest.mark.parametrize("precision", ["bf16x3", "fp16x3"])
@pytest.mark.parametrize("rows,n_ext,modes,bins", [(5000, 161, 1, 32), (20001, 40, 2, 33), (300, 3001, 4, 64)])
def test_sums_hold_every_pair(precision, rows, n_ext, modes, bins):
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    wl = synth.make_workload(n_int=rows, n_ext=n_ext, n_det=2, n_modes=modes, n_bins=bins, snr=0.1, seed=3, n_phi=4)
    ctx = dp.dotpe_create(0)
    try:
        bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m)
        for _ in range(5):
            eid = dp.dotpe_event_submit(ctx, bid, 0, rows, wl.event.psd, wl.event.data, wl.ext.t, wl.ext.R, n_phi=4,
                                        u_min=wl.event.u_min, precision=precision, flags=dp.DOTPE_FLAG_STORE_LNL)
            dp.dotpe_event_wait(ctx, eid, 60.0)
            ev = dp.dotpe_evidence(ctx, eid)
            lnl, row, col = (dp.dotpe_lnl_blocks(ctx, eid, 0, rows, 0, n_ext, what=w)
                             for w in (dp.DOTPE_LNL_MARG, dp.DOTPE_ROW_MARGINAL, dp.DOTPE_COL_MARGINAL))
            dp.dotpe_event_release(ctx, eid)
            assert np.max(np.abs(lnl)) < 50.0
            lp = lnl.astype(np.float64) + np.log(4.0)
            assert np.max(np.abs(row - _lse(lp, 1))) <= 5e-5
            assert np.max(np.abs(col - _lse(lp, 0))) <= 5e-5
            assert abs(ev["ln_z"] - (_lse(lp) - np.log(rows) - np.log(n_ext) - np.log(4))) <= 5e-5
    finally:
        dp.dotpe_destroy(ctx)
