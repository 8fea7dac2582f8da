"""More kinds of batches on one slot than the context keeps executable graphs for: each is
captured again when its turn comes, and the events' results stay the same bits."""
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_more_batch_shapes_than_kept_graphs():
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    wl = synth.make_workload(n_int=700, n_ext=70, n_det=2, n_modes=2, n_bins=32, snr=12.0, seed=4, n_phi=8)
    ctx = dp.dotpe_create(0, n_slots=1)
    try:
        bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m)
        call = dict(bank_id=bid, i0=0, i1=700, psd=wl.event.psd, data=wl.event.data, t=wl.ext.t, R=wl.ext.R, n_phi=8,
                    u_min=wl.event.u_min, precision="mixed", cut_delta=20.0)
        ref = None
        for n in list(range(1, 13)) * 2:
            for eid in dp.dotpe_batch_submit(ctx, [call] * n):
                dp.dotpe_event_wait(ctx, eid, 60.0)
                ev = dp.dotpe_evidence(ctx, eid)
                dp.dotpe_event_release(ctx, eid)
                ref = ref or ev
                assert (ev["ln_z"], ev["n_marginalised"]) == (ref["ln_z"], ref["n_marginalised"])
    finally:
        dp.dotpe_destroy(ctx)
