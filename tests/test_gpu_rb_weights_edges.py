"""Relative-binning weights where the kernel's blocks change: intervals of one point, of one
block of 512 points and one more, a thread count (128) and one more, the first and last
nodes, one to eight components, with and without arrival times.

Tolerance, before any run: FP64 rounding, 1e-11 of the largest weight, as for the paper's
binning.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dpx():
    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    ctx = dp.dotpe_create(0)
    yield dp, ctx
    dp.dotpe_destroy(ctx)


@pytest.mark.parametrize("comps", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("steps,lead,tail", [
    ((1,), 0, 0), ((1, 1, 1), 0, 3), ((512, 513, 1), 5, 0), ((127, 128, 129, 2), 0, 7), ((1025, 3, 511), 2, 2)])
@pytest.mark.parametrize("n_det", [1, 3])
def test_intervals_against_oracle(dpx, comps, steps, lead, tail, n_det):
    dp, ctx = dpx
    rng = np.random.default_rng(comps * 100 + len(steps))
    nodes = lead + np.concatenate([[0], np.cumsum(steps)]).astype(np.int64)
    N = int(nodes[-1]) + 1 + tail
    f = 20.0 + 0.25 * np.arange(N)
    df = rng.uniform(0.1, 0.3, N)
    psd = rng.uniform(0.5, 2.0, (n_det, N))
    data = rng.standard_normal((n_det, N)) + 1j * rng.standard_normal((n_det, N))
    # components of modulus 0.5 to 2: no division by a vanishing reference
    h0 = rng.uniform(0.5, 2.0, (comps, N)) * np.exp(2j * np.pi * rng.uniform(size=(comps, N)))
    for t0 in (rng.uniform(-0.02, 0.02, n_det), None):
        w_dh, w_hh = oracle.rb_weights(f, df, psd, data, h0, nodes, t0)
        g_dh, g_hh = dp.dotpe_rb_weights(ctx, f, df, psd, data, h0, nodes, t0)
        assert np.max(np.abs(g_dh - w_dh)) <= 1e-11 * np.max(np.abs(w_dh))
        assert np.max(np.abs(g_hh - w_hh)) <= 1e-11 * np.max(np.abs(w_hh))
