"""The tuner's choice is made per kind of launch: an event that may only take 32-sample tiles
does not leave its choice to the screened events of the same shape.

The screen's counters tell the tile form: 64-sample tiles count candidates that they do not
evaluate, 32-sample tiles evaluate every pair they count.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [dict(cut_delta=0.0), dict(cut_delta=20.0, flags="store")])
def test_a_narrow_event_does_not_choose_for_wide_ones(first):
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    rows, ext = 30000, 2048
    wl = synth.make_workload(n_int=rows, n_ext=ext, n_det=3, n_modes=4, n_bins=512, snr=15.0, seed=6)
    first = dict(first)
    if first.get("flags"):
        first["flags"] = dp.DOTPE_FLAG_STORE_LNL
    counts = {}
    for name, calls in (("alone", [{}]), ("after", [first, {}])):
        ctx = dp.dotpe_create(0, flags=dp.DOTPE_CONFIG_AUTOTUNE)
        try:
            bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m)
            for c in calls:
                kw = dict(cut_delta=20.0)
                kw.update(c)
                eid = dp.dotpe_event_submit(ctx, bid, 0, rows, wl.event.psd, wl.event.data, wl.ext.t, wl.ext.R,
                                            u_min=wl.event.u_min, precision="mixed", **kw)
                dp.dotpe_event_wait(ctx, eid, 60.0)
                ev = dp.dotpe_evidence(ctx, eid)
                dp.dotpe_event_release(ctx, eid)
            counts[name] = (ev["n_screen_candidates"], ev["n_screen_evaluated"])
        finally:
            dp.dotpe_destroy(ctx)
    cand, done = counts["alone"]
    assert cand > done > 0  # (this shape is faster in 64-sample tiles)
    cand, done = counts["after"]
    assert cand > done > 0
