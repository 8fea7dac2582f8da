"""The coherent-ML cut keeps the same phases however an event's pairs are evaluated: with and
without stored values, on phase grids that are and are not evaluated four phases at a time,
alone and in a batch.

The kept set is compared exactly: n_marginalised, the finite entries of the samples'
marginals, and for stored values ln Lbar finite just where ln L^ML reaches the threshold.
Tolerance of the marginals, before any run: both sum the same FP32 terms in another order,
~2e-6 of ln P plus the FP32 rounding of a value below 128 (4e-6 each): 2e-5.  Some
phases lie within FP32 rounding of the threshold in these events.
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


def _read(dp, ctx, eid, rows, n_ext, store):
    dp.dotpe_event_wait(ctx, eid, 60.0)
    ev = dp.dotpe_evidence(ctx, eid)
    col = dp.dotpe_lnl_blocks(ctx, eid, 0, 1, 0, n_ext, what=dp.DOTPE_COL_MARGINAL)
    pairs = [dp.dotpe_lnl_blocks(ctx, eid, 0, rows, 0, n_ext, what=w)
             for w in (dp.DOTPE_LNL_MARG, dp.DOTPE_LNL_ML_MAX)] if store else None
    dp.dotpe_event_release(ctx, eid)
    return ev, col, pairs


@pytest.mark.parametrize("rows,n_ext,n_phi,modes", [(20000, 1500, 32, 4), (30000, 700, 64, 3), (20000, 900, 30, 4),
                                                    (20000, 900, 128, 2)])
@pytest.mark.parametrize("above", [4.0, 8.0])
def test_the_kept_phases_do_not_depend_on_the_route(dpx, rows, n_ext, n_phi, modes, above):
    dp, ctx = dpx
    wl = synth.make_workload(n_int=rows, n_ext=n_ext, n_det=3, n_modes=modes, n_bins=64, snr=8.0, seed=5 + n_phi,
                             n_phi=n_phi)
    bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m)
    call = dict(bank_id=bid, i0=0, i1=rows, psd=wl.event.psd, data=wl.event.data, t=wl.ext.t, R=wl.ext.R,
                n_phi=n_phi, u_min=wl.event.u_min, precision="mixed")
    # a cut that leaves the phases from ln L^ML of about 4 (millions) or 8 on
    best = _read(dp, ctx, dp.dotpe_event_submit(ctx, cut_delta=1.0, **call), rows, n_ext, False)[0]["max_lnl_ml"]
    call.update(cut_delta=best - above)
    ev0, col0, (lnl, ml) = _read(dp, ctx, dp.dotpe_event_submit(ctx, flags=dp.DOTPE_FLAG_STORE_LNL, **call), rows,
                                 n_ext, True)
    got = [_read(dp, ctx, dp.dotpe_event_submit(ctx, **call), rows, n_ext, False)]
    got += [_read(dp, ctx, eid, rows, n_ext, False) for eid in dp.dotpe_batch_submit(ctx, [call, call])]
    dp.dotpe_bank_release(ctx, bid)
    assert np.all(ml[np.isfinite(lnl)] >= np.float32(ev0["lnl_ml_threshold"]))
    assert ev0["n_marginalised"] > (100000 if above == 4.0 else 1000)
    for ev, col, _ in got:
        assert ev["n_marginalised"] == ev0["n_marginalised"]
        assert np.array_equal(np.isfinite(col), np.isfinite(col0))
        ok = np.isfinite(col)
        assert np.max(np.abs(col[ok] - col0[ok])) <= 2e-5
