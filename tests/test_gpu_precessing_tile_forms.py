"""The screen of a polarisation-resolved bank in its three tile forms: 64-sample tiles on CTA
pairs (the default for large events), on one SM each, and 32-sample tiles.  Ragged rows and samples, an odd
number of 32-sample tiles and of bank tiles, a shape large enough for pilot tiles, one to
four modes and one to three detectors, odd k-blocks.

Tolerances, before any run: all forms mark the same tiles and refine them alike, so counts
and arguments are equal and ln Z agrees to 1e-9, as for mode banks; ln Z between the
oracle's cut and uncut values within 1e-2, or within 1e-2 of the FP32 path at the largest
shape.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def forms():
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    ctxs = [dp.dotpe_create(0, flags=f) for f in (0, dp.DOTPE_CONFIG_SINGLE_CTA_TILES, dp.DOTPE_CONFIG_NARROW_TILES)]
    yield dp, ctxs
    for c in ctxs:
        dp.dotpe_destroy(c)


def _run(dp, ctx, wl, precision):
    I = wl.bank.h.shape[0]
    bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m, wl.bank.ln_w)
    try:
        eid = dp.dotpe_event_submit(ctx, bid, 0, I, wl.event.psd, wl.event.data, wl.ext.t, None, wl.ext.ln_w,
                                    n_phi=wl.event.n_phi, u_min=wl.event.u_min, cut_delta=20.0, precision=precision,
                                    F=wl.ext.F)
        dp.dotpe_event_wait(ctx, eid, 60.0)
        ev = dp.dotpe_evidence(ctx, eid)
        dp.dotpe_event_release(ctx, eid)
    finally:
        dp.dotpe_bank_release(ctx, bid)
    return ev


@pytest.mark.parametrize("shape", [(1, 1, 3, 4, 64), (129, 33, 1, 1, 96), (300, 77, 2, 3, 128), (513, 97, 3, 2, 200),
                                   (257, 128, 3, 4, 250), (2100, 1000, 3, 4, 128),
                                   # enough work for the 64-sample tiles (the shapes above stay narrow)
                                   (4033, 2017, 3, 4, 490), (6200, 2399, 2, 2, 510), (8201, 3521, 1, 1, 512)],
                         ids=lambda s: "x".join(map(str, s)))
def test_forms_agree(forms, shape):
    import oracle
    dp, ctxs = forms
    I, E, D, M, B = shape
    wl = synth.make_precessing_workload(I, E, D, M, B, snr=14.0, seed=I + E, n_phi=32, ln_w="random")
    pair, one, narrow = (_run(dp, c, wl, "mixed") for c in ctxs)
    for k in ("n_refined_tiles", "arg_i", "arg_e", "arg_o", "ln_z", "max_lnl_ml", "n_eff", "n_marginalised"):
        assert pair[k] == one[k], k
    for k in ("n_refined_tiles", "arg_i", "arg_e", "arg_o", "max_lnl_ml"):
        assert pair[k] == narrow[k], k
    assert pair["ln_z"] == pytest.approx(narrow["ln_z"], abs=1e-9)
    if I * E > 300000:
        ref = _run(dp, ctxs[0], wl, "fp32")
        assert abs(pair["ln_z"] - ref["ln_z"]) <= 1e-2
        assert pair["max_lnl_ml"] == pytest.approx(ref["max_lnl_ml"], abs=1e-3)
        return
    P = oracle.OracleProblem(wl.bank, wl.ext, wl.event)
    lo, hi = (P.evidence(P.eval_grid(c)[0])["ln_z"] for c in (20.0, 0.0))
    assert lo - 1e-2 <= pair["ln_z"] <= hi + 1e-2
