"""Batches whose events fall on both sides of the line from which an event launches its own
kernels (96 tiles of 128 x 32 pairs per SM): the results of every event are those it has alone,
in mixed batches, in batches of one kind only, replayed, and without graphs.

Tolerance, before any run: the same kernels' products in another launch form, so the values an
event has alone to 1e-6 in ln Z and max ln L^ML, and the same refined tiles and maximum.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("precision,cut", [("mixed", 20.0), ("fp16x3", 0.0)])
def test_events_of_a_batch_equal_events_alone(graphs, precision, cut):
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    ctx = dp.dotpe_create(0, flags=0 if graphs else dp.DOTPE_CONFIG_NO_GRAPHS)
    try:
        n_sms = dp.dotpe_device_info(ctx)[0]
        rows = 16384
        large = 32 * ((96 * n_sms + rows // 128 - 1) // (rows // 128)) - 7  # just past the line
        rng = np.random.default_rng(5)
        bank = synth.make_bank(rng, rows, 2, 24)
        bid = dp.dotpe_bank_load(ctx, bank.h, bank.f, bank.w, bank.mode_m, bank.ln_w)
        specs = []
        for n_ext, n_det in ((large, 2), (100, 3), (large - 64, 3), (33, 2), (large + 40, 3)):
            ext = synth.make_extrinsic(rng, n_ext, n_det, bank)
            ev = synth.make_event(rng, bank, ext, n_det, snr=14.0, n_phi=8)
            specs.append(dict(bank_id=bid, i0=0, i1=rows, psd=ev.psd, data=ev.data, t=ext.t, R=ext.R, n_phi=8,
                              u_min=ev.u_min, cut_delta=cut, precision=precision))

        def read(eid):
            dp.dotpe_event_wait(ctx, eid, 120.0)
            e = dp.dotpe_evidence(ctx, eid)
            dp.dotpe_event_release(ctx, eid)
            return e

        alone = [read(dp.dotpe_event_submit(ctx, **s)) for s in specs]
        for pick in ((0, 1, 2, 3, 4), (0, 1, 2, 3, 4), (0, 4), (1, 3), (2,), (3, 0)):
            for k, eid in zip(pick, dp.dotpe_batch_submit(ctx, [specs[k] for k in pick])):
                e = read(eid)
                assert abs(e["ln_z"] - alone[k]["ln_z"]) <= 1e-6, (pick, k)
                assert abs(e["max_lnl_ml"] - alone[k]["max_lnl_ml"]) <= 1e-6, (pick, k)
                for q in ("arg_i", "arg_e", "arg_o", "n_refined_tiles", "device_status"):
                    assert e[q] == alone[k][q], (pick, k, q)
        dp.dotpe_bank_release(ctx, bid)
    finally:
        dp.dotpe_destroy(ctx)
