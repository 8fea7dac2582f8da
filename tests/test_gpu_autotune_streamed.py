"""Screened events streamed in blocks of different rows in a context with the tuner on: every
block is refined with its own <h|h> bound, or none, whichever tile form the tuner takes.  Few
samples leave half of a 64-sample tile empty, so that the tuner takes 32-sample tiles.

Tolerance, before any run: the refined pairs and kept phases are the same, sums in another
order at most, ~2e-6 of ln P plus its FP32 rounding below 256 (1.5e-5 each): 4e-5.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ext", [5, 32, 40, 300])
def test_streamed_events_in_a_tuned_context(n_ext):
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    rows, block = 40000, 8192
    wl = synth.make_workload(n_int=rows, n_ext=n_ext, n_det=3, n_modes=4, n_bins=128, snr=18.0, seed=31 + n_ext)
    # rows of very different norms from block to block (the bound's scale follows them)
    wl.bank.h *= np.repeat([1.0, 0.02, 3.0, 0.3, 1.0], block)[:rows, None, None]
    out = []
    for flags in (0, dp.DOTPE_CONFIG_AUTOTUNE):
        ctx = dp.dotpe_create(0, flags=flags)
        try:
            bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m)
            for _ in range(2):  # tuned on the first, from the cache on the second
                eid = dp.dotpe_event_submit(ctx, bid, 0, rows, wl.event.psd, wl.event.data, wl.ext.t, wl.ext.R,
                                            u_min=wl.event.u_min, precision="mixed", cut_delta=20.0, block_rows=block)
                dp.dotpe_event_wait(ctx, eid, 60.0)
                out.append((dp.dotpe_evidence(ctx, eid),
                            dp.dotpe_lnl_blocks(ctx, eid, 0, rows, 0, 1, what=dp.DOTPE_ROW_MARGINAL),
                            dp.dotpe_lnl_blocks(ctx, eid, 0, 1, 0, n_ext, what=dp.DOTPE_COL_MARGINAL)))
                dp.dotpe_event_release(ctx, eid)
        finally:
            dp.dotpe_destroy(ctx)
    ev0, row0, col0 = out[0]
    assert ev0["n_marginalised"] > 0
    for ev, row, col in out[1:]:
        assert ev["n_marginalised"] == ev0["n_marginalised"]
        for a, b in ((row, row0), (col, col0)):
            ok = np.isfinite(b)
            assert np.array_equal(np.isfinite(a), ok)
            assert np.max(np.abs(a[ok] - b[ok])) <= 4e-5
        assert abs(ev["ln_z"] - ev0["ln_z"]) <= 4e-5
