"""Pre-selection's choice of rows around its blocks of 2,048: the rows kept, their order and
the row of the maximum against the returned ln L^inco.ML (the same FP64 values: exact)."""
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


@pytest.mark.parametrize("rows", [1, 7, 255, 2047, 2048, 2049, 4096, 6151])
@pytest.mark.parametrize("repeat", [False, True])
def test_selection_is_exact(dpx, rows, repeat):
    dp, ctx = dpx
    wl = synth.make_workload(n_int=rows, n_ext=2, n_det=2, n_modes=2, n_bins=48, snr=12.0, seed=rows)
    h = np.repeat(wl.bank.h[:1], rows, axis=0) if repeat else wl.bank.h  # repeat: every row attains the maximum
    ps = synth.make_presel_inputs(wl, n_t=20, dt=1.5e-3, seed=rows + 1)
    pol = np.repeat(ps.pol[:1], rows, axis=0) if repeat else ps.pol
    bid = dp.dotpe_bank_load(ctx, h, wl.bank.f, wl.bank.w, wl.bank.mode_m, wl.bank.ln_w, pol=pol)
    try:
        for delta in (0.0, 2.0, 20.0, 1e6):
            r = dp.dotpe_preselect(ctx, bid, 0, rows, wl.event.psd, wl.event.data, ps.t_grid, n_phi=8, delta=delta,
                                   precision="fp16x3")
            inco = np.asarray(r["lnl_inco"])
            assert r["max_lnl_inco"] == inco.max() and r["arg_i"] == int(np.argmax(inco))
            assert np.array_equal(r["selected"], np.nonzero(inco >= inco.max() - delta)[0])
    finally:
        dp.dotpe_bank_release(ctx, bid)
