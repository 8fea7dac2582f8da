"""Stage times of a batch whose events launch their own kernels: an event's refinement time is
its own, not the kernels of the events behind it.

Two equal events: their screens and refinements are the same work, one after the other.  The
refinement is a small part of the screen here, so that a time that held the other event's
screen would be several times as long; allowed, before any run: twice the other's and 50 us.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_refinement_time_is_the_events_own():
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    rows, ext = 65536, 1024  # 512 x 32 tiles: more than 96 per SM
    wl = synth.make_workload(n_int=rows, n_ext=ext, n_det=2, n_modes=3, n_bins=128, snr=25.0, seed=14)
    ctx = dp.dotpe_create(0)
    try:
        assert 512 * 32 >= 96 * dp.dotpe_device_info(ctx)[0]
        bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m)
        call = dict(bank_id=bid, i0=0, i1=rows, psd=wl.event.psd, data=wl.event.data, t=wl.ext.t, R=wl.ext.R,
                    u_min=wl.event.u_min, precision="mixed", cut_delta=20.0)
        for _ in range(3):
            ids = dp.dotpe_batch_submit(ctx, [call, call])
            for eid in ids:
                dp.dotpe_event_wait(ctx, eid, 60.0)
            st = [dp.dotpe_event_poll(ctx, eid)[1] for eid in ids]
            for eid in ids:
                dp.dotpe_event_release(ctx, eid)
        first, second = (s["refine_ms"] for s in st)
        assert 0.0 < first <= 2.0 * second + 0.05
        assert all(s["refine_ms"] <= s["fused_ms"] <= s["device_ms"] for s in st)
    finally:
        dp.dotpe_destroy(ctx)
