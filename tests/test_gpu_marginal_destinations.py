"""dotpe_lnl_blocks' marginals into every kind of memory that a copy reaches: host, pinned
host, device, device memory that is not aligned to a float, managed memory.  The values are
the same bytes.
"""
import ctypes

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

ROWS, EXT = 333, 77


def test_marginals_reach_every_kind_of_memory():
    import torch

    import __graft_entry__ as ge
    ge.build()
    import paper_2507_16022_gb300 as dp
    wl = synth.make_workload(n_int=ROWS, n_ext=EXT, n_det=2, n_modes=2, n_bins=48, snr=10.0, seed=8, n_phi=8)
    rt = ctypes.CDLL("libcudart.so.13")
    ctx = dp.dotpe_create(0)
    managed = ctypes.c_void_p()
    assert rt.cudaMallocManaged(ctypes.byref(managed), ctypes.c_size_t(4096), 1) == 0
    try:
        bid = dp.dotpe_bank_load(ctx, wl.bank.h, wl.bank.f, wl.bank.w, wl.bank.mode_m)
        eid = dp.dotpe_event_submit(ctx, bid, 0, ROWS, wl.event.psd, wl.event.data, wl.ext.t, wl.ext.R, n_phi=8,
                                    u_min=wl.event.u_min, precision="fp16x3")
        dp.dotpe_event_wait(ctx, eid, 60.0)

        def into(what, n, ptr):
            a = (0, n, 0, 1) if what == dp.DOTPE_ROW_MARGINAL else (0, 1, 0, n)
            assert dp.load().dotpe_lnl_blocks(ctx, ctypes.c_uint64(eid), *map(ctypes.c_int64, a), what,
                                              ctypes.c_void_p(ptr), ctypes.c_int64(n)) == 0

        for what, n in ((dp.DOTPE_ROW_MARGINAL, ROWS), (dp.DOTPE_COL_MARGINAL, EXT)):
            ref = np.empty(n, np.float32)
            into(what, n, ref.ctypes.data)
            assert np.all(np.isfinite(ref))
            pinned = torch.empty(n, dtype=torch.float32, pin_memory=True)
            into(what, n, pinned.data_ptr())
            assert pinned.numpy().tobytes() == ref.tobytes()
            for off in (0, 4, 2, 1):
                dev = torch.zeros(4 * n + 8, dtype=torch.uint8, device="cuda")
                torch.cuda.synchronize()
                into(what, n, dev.data_ptr() + off)
                got = dev.cpu().numpy()
                assert got[off:off + 4 * n].tobytes() == ref.tobytes()
                assert not got[:off].any() and not got[off + 4 * n:].any()
            into(what, n, managed.value)
            torch.cuda.synchronize()
            assert ctypes.string_at(managed.value, 4 * n) == ref.tobytes()
    finally:
        rt.cudaFree(managed)
        dp.dotpe_destroy(ctx)
