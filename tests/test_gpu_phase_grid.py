"""The marginalising epilogue over phase grids, mode sets and cuts where its paths change:
grids that are and are not multiples of four phases, of one and of several mask words, banks
whose azimuthal numbers leave gaps, dense tiles (every lane evaluates its own pair) and
sparse ones (collected pairs, four lanes each).

Tolerances, before any run: |d ln Lbar| and |d ln L^ML| <= 1e-3 per pair, the split
precisions' bound.  Stored and not stored runs of one event evaluate the same pairs with
the same thresholds, apart from roundings of ~1e-7 ln L^ML in the phase sums: |d ln Z| <=
1e-4 and |d max ln L^ML| <= 1e-4.
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


def _event(dp, ctx, bid, wl, n_phi, cut, precision, store):
    I, E = wl.bank.h.shape[0], wl.ext.t.shape[0]
    eid = dp.dotpe_event_submit(ctx, bid, 0, I, wl.event.psd, wl.event.data, wl.ext.t, wl.ext.R, wl.ext.ln_w,
                                n_phi=n_phi, u_min=wl.event.u_min, cut_delta=cut, precision=precision,
                                flags=dp.DOTPE_FLAG_STORE_LNL if store else 0)
    dp.dotpe_event_wait(ctx, eid, 60.0)
    out = [dp.dotpe_evidence(ctx, eid)]
    if store:
        out += [dp.dotpe_lnl_blocks(ctx, eid, 0, I, 0, E, w) for w in (dp.DOTPE_LNL_MARG, dp.DOTPE_LNL_ML_MAX)]
    dp.dotpe_event_release(ctx, eid)
    return out


@pytest.mark.parametrize("n_phi", [1, 3, 4, 30, 32, 33, 64, 126, 128])
@pytest.mark.parametrize("mode_m", [(2,), (1, 3), (2, 3, 4), (1, 2, 3, 4)])
def test_phase_grids_against_oracle(dpx, n_phi, mode_m):
    dp, ctx = dpx
    wl = synth.make_workload(n_int=131, n_ext=34, n_det=2, n_modes=len(mode_m), n_bins=65, snr=12.0,
                             seed=40 + n_phi, n_phi=n_phi, ln_w="random")
    wl.bank.mode_m = np.array(mode_m, dtype=np.int32)
    ref, _ = oracle.OracleProblem(wl.bank, wl.ext, wl.event).eval_grid(0.0)
    bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m, wl.bank.ln_w)
    try:
        for precision in ("fp32", "fp16x3", "bf16x3"):
            _, lnl, ml = _event(dp, ctx, bid, wl, n_phi, 0.0, precision, True)
            assert np.max(np.abs(lnl - ref["lnl_marg"])) <= 1e-3, precision
            assert np.max(np.abs(ml - ref["lnl_ml_max"])) <= 1e-3, precision
            # with a cut every pair's best ln L^ML is still stored
            _, _, ml = _event(dp, ctx, bid, wl, n_phi, 8.0, precision, True)
            assert np.max(np.abs(ml - ref["lnl_ml_max"])) <= 1e-3, precision
    finally:
        dp.dotpe_bank_release(ctx, bid)


@pytest.mark.parametrize("n_phi", [5, 32, 34, 128])
@pytest.mark.parametrize("cut", [2.0, 12.0, 200.0])  # few pairs of a tile left, some, all
@pytest.mark.parametrize("n_det", [1, 3])
def test_collected_pairs_match_stored_ones(dpx, n_phi, cut, n_det):
    dp, ctx = dpx
    wl = synth.make_workload(n_int=389, n_ext=97, n_det=n_det, n_modes=4, n_bins=96, snr=14.0, seed=7, n_phi=n_phi,
                             ln_w="random")
    bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m, wl.bank.ln_w)
    try:
        # mixed: the refinement's threshold is frozen, so both runs keep the same pairs
        a = _event(dp, ctx, bid, wl, n_phi, cut, "mixed", True)[0]
        b = _event(dp, ctx, bid, wl, n_phi, cut, "mixed", False)[0]
        assert abs(a["ln_z"] - b["ln_z"]) <= 1e-4
        assert abs(a["max_lnl_ml"] - b["max_lnl_ml"]) <= 1e-4
        assert (a["arg_i"], a["arg_e"]) == (b["arg_i"], b["arg_e"])
    finally:
        dp.dotpe_bank_release(ctx, bid)
