"""Blocks recomputed into device memory, with the next calls on the context's heels: the
values are the bytes that a host destination gets.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp16x3", "mixed"])
def test_recomputed_blocks_into_device_memory(precision):
    import torch

    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    rows, ext = 3000, 700
    wl = synth.make_workload(n_int=rows, n_ext=ext, n_det=2, n_modes=3, n_bins=64, snr=12.0, seed=12, n_phi=8)
    ctx = dp.dotpe_create(0)
    try:
        bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m)

        def event():
            return dp.dotpe_event_submit(ctx, bid, 0, rows, wl.event.psd, wl.event.data, wl.ext.t, wl.ext.R, n_phi=8,
                                         u_min=wl.event.u_min, precision=precision)

        eid = event()
        dp.dotpe_event_wait(ctx, eid, 60.0)
        blocks = [(0, rows, 0, ext), (0, rows, 1, ext), (100, 2900, 0, 650)]
        ref = [dp.dotpe_lnl_blocks(ctx, eid, *b) for b in blocks]
        outs, others = [], []
        for b in blocks:
            out = torch.empty(b[1] - b[0], b[3] - b[2], dtype=torch.float32, device="cuda")
            outs.append(dp.dotpe_lnl_blocks(ctx, eid, *b, out=out))
            others.append(event())
        for o in others:
            dp.dotpe_event_wait(ctx, o, 60.0)
        for r, o in zip(ref, outs):
            assert np.array_equal(r, o.cpu().numpy())
    finally:
        dp.dotpe_destroy(ctx)
