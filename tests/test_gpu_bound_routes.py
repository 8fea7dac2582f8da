"""A screened event's results do not depend on whether its screen had the tensor-core <h|h>
bound: with it, in a context of 32-sample tiles (none), in a context whose budget has no room
for it, and in a batch, the same bits.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

KEYS = ("ln_z", "n_eff", "n_eff_int", "n_eff_ext", "max_lnl_ml", "arg_i", "arg_e", "arg_o", "n_marginalised",
        "n_refined_tiles", "lnl_ml_threshold")
ROWS, EXT, KPAD = 20000, 1500, 128


@pytest.mark.parametrize("snr,cut", [(8.0, 24.0), (8.0, 20.0), (14.0, 20.0)])  # dense, between, sparse tiles
@pytest.mark.parametrize("modes", [2, 4])
def test_results_do_not_depend_on_the_bound(snr, cut, modes):
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    wl = synth.make_workload(n_int=ROWS, n_ext=EXT, n_det=3, n_modes=modes, n_bins=KPAD // 2, snr=snr, seed=77,
                             ln_w="random")
    foot = {}

    def run(name, batch=False, **cfg):
        ctx = dp.dotpe_create(0, **cfg)
        try:
            bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m, wl.bank.ln_w)
            call = dict(bank_id=bid, i0=0, i1=ROWS, psd=wl.event.psd, data=wl.event.data, t=wl.ext.t, R=wl.ext.R,
                        ln_w_ext=wl.ext.ln_w, u_min=wl.event.u_min, precision="mixed", cut_delta=cut)
            ids = dp.dotpe_batch_submit(ctx, [call] * 2) if batch else [dp.dotpe_event_submit(ctx, **call)]
            out = []
            for eid in ids:
                dp.dotpe_event_wait(ctx, eid, 60.0)
                foot[name] = dp.dotpe_event_poll(ctx, eid)[1]["footprint_bytes"]
                ev = dp.dotpe_evidence(ctx, eid)
                out.append([ev[k] for k in KEYS] +
                           [dp.dotpe_lnl_blocks(ctx, eid, 0, ROWS, 0, 1, what=dp.DOTPE_ROW_MARGINAL),
                            dp.dotpe_lnl_blocks(ctx, eid, 0, 1, 0, EXT, what=dp.DOTPE_COL_MARGINAL)])
                dp.dotpe_event_release(ctx, eid)
            return out
        finally:
            dp.dotpe_destroy(ctx)

    ref = run("bound")[0]
    assert ref[KEYS.index("n_marginalised")] > 0
    got = run("narrow", flags=dp.DOTPE_CONFIG_NARROW_TILES) + run("batch", batch=True)
    bound = foot["bound"] - foot["narrow"]
    assert bound >= ROWS * EXT * 2
    bank = 12 * modes * ROWS * KPAD + (1 << 20)
    got += run("tight", hbm_budget_bytes=bank + foot["narrow"] + bound // 2)
    assert foot["tight"] == foot["narrow"]
    for out in got:
        for k, a, b in zip(KEYS + ("row", "col"), out, ref):
            assert np.array_equal(a, b), k
