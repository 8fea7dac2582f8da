"""Events of the split precisions with a running cut, nothing stored: the threshold rises
while the tiles are evaluated, from none at all in the first ones.

Tolerance, before any run: with a cut of 40 below a best ln L^ML of about 110 the dropped
phases hold less than e^-25 of the evidence, so ln Z is that of the event without a cut up
to the FP32 sums: 1e-4.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16x3", "fp16x3"])
@pytest.mark.parametrize("rows,n_ext,modes", [(20001, 97, 2), (1500, 2050, 4)])
def test_running_cut_keeps_the_evidence(precision, rows, n_ext, modes):
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    wl = synth.make_workload(n_int=rows, n_ext=n_ext, n_det=3, n_modes=modes, n_bins=64, snr=15.0, seed=21, n_phi=16,
                             insert_injection=True)
    ctx = dp.dotpe_create(0)
    try:
        bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m)

        def event(cut):
            eid = dp.dotpe_event_submit(ctx, bid, 0, rows, wl.event.psd, wl.event.data, wl.ext.t, wl.ext.R, n_phi=16,
                                        u_min=wl.event.u_min, precision=precision, cut_delta=cut)
            dp.dotpe_event_wait(ctx, eid, 60.0)
            ev = dp.dotpe_evidence(ctx, eid)
            dp.dotpe_event_release(ctx, eid)
            return ev

        ref = event(0.0)
        assert ref["max_lnl_ml"] > 80.0
        for _ in range(10):
            ev = event(40.0)
            assert abs(ev["ln_z"] - ref["ln_z"]) <= 1e-4
            assert ev["max_lnl_ml"] == pytest.approx(ref["max_lnl_ml"], abs=1e-3)
            assert 0 < ev["n_marginalised"] < ref["n_marginalised"]
    finally:
        dp.dotpe_destroy(ctx)
