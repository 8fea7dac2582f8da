"""The FP32 pre-selection of polarisation-resolved banks at the edges of its blocks: rows
around a block's four, times around a thread's two (16 apart), a warp's 32 and a pass's 128,
bins around the operand's groups of four and the chunks of 32, one to four modes, with
component weights (the weighted rows) and with the plain quadrature.

Tolerance, before any run: the pre-selection's 2e-3 + 1e-4 ln L^ML per (row, detector)
against the oracle.
"""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("rows,n_t,bins,modes,n_phi", [
    (1, 1, 33, 1, 1), (3, 15, 34, 2, 8), (4, 16, 63, 3, 31), (5, 17, 64, 4, 32), (9, 33, 65, 4, 32),
    (13, 100, 97, 3, 16), (6, 127, 40, 4, 32), (7, 128, 41, 2, 32), (8, 129, 42, 4, 5), (11, 200, 67, 4, 32)])
@pytest.mark.parametrize("weights", [True, False])
def test_edges_against_oracle(dpx, rows, n_t, bins, modes, n_phi, weights):
    dp, ctx = dpx
    rw = synth.make_rb_workload(rows, 4, 2, modes, bins, n_fine=16384, snr=12.0, seed=rows + bins, precessing=True)
    w = oracle.rb_weights(rw.f_fine, rw.dff, rw.psd_fine, rw.data_fine, rw.h0_fine, rw.nodes, rw.t0) if weights else None
    t_grid = rw.t0[:, None] + (np.arange(n_t) - n_t // 2)[None, :] * 5e-4
    ref = oracle.PreselProblem(rw.bank.f, rw.bank.w, rw.bank.mode_m, rw.bank.h, None, rw.event.psd, rw.event.data,
                               t_grid, n_phi=n_phi, rb=w).run(delta=20.0)
    bid = dp.dotpe_bank_load(ctx, rw.bank.h, rw.bank.f, rw.bank.w, rw.bank.mode_m, rw.bank.ln_w)
    try:
        psd, data = (None, None) if weights else (rw.event.psd, rw.event.data)
        r = dp.dotpe_preselect(ctx, bid, 0, rows, psd, data, t_grid, n_phi=n_phi, delta=20.0, precision="fp32", rb=w)
    finally:
        dp.dotpe_bank_release(ctx, bid)
    assert np.all(np.abs(r["lnl_ml"] - ref["ml"]) <= 2e-3 + 1e-4 * np.abs(ref["ml"]))
    o, t = r["arg_ot"][..., 0], r["arg_ot"][..., 1]
    assert np.all((0 <= o) & (o < n_phi) & (0 <= t) & (t < n_t))
