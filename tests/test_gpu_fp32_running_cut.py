"""FP32 events with a cut: what is in flight before a maximum is known is marginalised whole,
two blocks of 64 x 32 pairs per SM whatever the number of modes; the rest is cut.

The reference count is the mixed event's, whose threshold is final before it marginalises;
the FP32 event keeps those phases (to the ~1e-3 of them within the two products' differences
at the threshold) and at most what its first blocks hold besides; allowed, before any run:
10% more for thresholds that are still rising.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("modes", [1, 2, 3, 4])
def test_only_the_first_blocks_go_uncut(modes):
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    rows, n_ext, n_phi = 12000, 200, 16
    wl = synth.make_workload(n_int=rows, n_ext=n_ext, n_det=2, n_modes=modes, n_bins=96, snr=16.0, seed=9, n_phi=n_phi,
                             insert_injection=True)
    ctx = dp.dotpe_create(0)
    try:
        n_sms = dp.dotpe_device_info(ctx)[0]
        bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m)
        ev = {}
        for precision in ("mixed", "fp32"):
            eid = dp.dotpe_event_submit(ctx, bid, 0, rows, wl.event.psd, wl.event.data, wl.ext.t, wl.ext.R, n_phi=n_phi,
                                        u_min=wl.event.u_min, precision=precision, cut_delta=20.0)
            dp.dotpe_event_wait(ctx, eid, 60.0)
            ev[precision] = dp.dotpe_evidence(ctx, eid)
            dp.dotpe_event_release(ctx, eid)
        first = 2 * n_sms * 64 * 32 * n_phi
        assert first < 0.6 * rows * n_ext * n_phi
        kept, least = ev["fp32"]["n_marginalised"], ev["mixed"]["n_marginalised"]
        assert 0.999 * least <= kept <= 1.1 * (first + least)
    finally:
        dp.dotpe_destroy(ctx)
