"""Posterior draws at the edges of the draw's blocks: one row or sample, row counts around the
256-row blocks of the row weights, extrinsic counts around the 32-entry steps, uniforms at the
ends of [0, 1).  (Events without a cut: with one, a running maximum keeps pairs by an earlier
threshold, and a draw that falls on one of those is refused by the call.)

The extrinsic draw is repeated in FP64 from the event's own stored values: the same index, or a
uniform within 1e-12 of the boundary between the two (sums in another order).  The row draw is
repeated from the row marginals that the ABI hands out in FP32 (1.2e-7 relative in a logarithm
of order 100: 1.2e-5 in a weight), so a uniform within 1e-4 of a boundary may go either way.
"""
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


def pick(lnw, u, tol):
    """(index, indices a uniform within tol of u could take) for weights exp(lnw)."""
    w = np.exp(lnw - lnw.max())
    c = np.cumsum(w)
    t = c[-1]
    at = lambda x: int(np.searchsorted(c, min(x * t, np.nextafter(t, 0.0)), side="right"))  # noqa: E731
    return at(u), range(at(max(0.0, u - tol)), at(u + tol) + 1), w


@pytest.mark.parametrize("n_int,n_ext", [(1, 1), (2, 31), (255, 32), (256, 33), (257, 64), (513, 65), (700, 129)])
@pytest.mark.parametrize("ln_w", ["zero", "random"])
def test_draws_from_the_events_own_weights(dpx, n_int, n_ext, ln_w):
    dp, ctx = dpx
    wl = synth.make_workload(n_int=n_int, n_ext=n_ext, n_det=2, n_modes=4, n_bins=70, snr=9.0, seed=n_int + n_ext,
                             n_phi=24, ln_w=ln_w)
    bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m, wl.bank.ln_w)
    lw = wl.ext.ln_w if ln_w == "random" else None
    try:
        eid = dp.dotpe_event_submit(ctx, bid, 0, n_int, wl.event.psd, wl.event.data, wl.ext.t, wl.ext.R, lw,
                                    n_phi=24, u_min=wl.event.u_min, cut_delta=0.0, precision="fp16x3",
                                    flags=dp.DOTPE_FLAG_STORE_LNL)
        dp.dotpe_event_wait(ctx, eid, 60.0)
        lnl = dp.dotpe_lnl_blocks(ctx, eid, 0, n_int, 0, n_ext).astype(np.float64)
        row = dp.dotpe_lnl_blocks(ctx, eid, 0, n_int, 0, n_ext, what=dp.DOTPE_ROW_MARGINAL).astype(np.float64)
        uni = np.random.default_rng(3).random((257, 4))
        uni[0], uni[1] = 0.0, 1.0 - 2.0 ** -53
        uni[2], uni[3] = [0.0, 1.0 - 2.0 ** -53] * 2, [1.0 - 2.0 ** -53, 0.0] * 2
        i, e, o, d = dp.dotpe_posterior_samples(ctx, eid, uni)
        dp.dotpe_event_release(ctx, eid)
    finally:
        dp.dotpe_bank_release(ctx, bid)
    assert np.all((0 <= o) & (o < 24)) and np.all(np.isfinite(d)) and np.all(d > 0)
    for s in range(uni.shape[0]):
        _, near, w = pick(row, uni[s, 0], 1e-4)
        assert i[s] in near and w[i[s]] > 0, s
        x = lnl[i[s]] + (0.0 if lw is None else lw)
        _, near, w = pick(x, uni[s, 1], 1e-12)
        assert e[s] in near and w[e[s]] > 0, s
