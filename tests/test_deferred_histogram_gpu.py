"""The deferred histogram's kernel queues the passing events of several tiles until
they fill a warp: no, few, nearly all events passing, one bin and many, counts
around the tiles and the grid, several chunks, against the per-event outputs."""
import numpy as np
import pytest
import torch

import paper_1002_3446_gb300 as tess

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pt_min,bins", [(0.01, 1), (0.01, 1024), (20.0, 7), (300.0, 40)])
@pytest.mark.parametrize("N,chunk", [(1, 0), (33, 0), (128 * 608 + 31, 0), (400_003, 0), (60_000, 1 << 20)])
def test_deferred_histogram(pt_min, bins, N, chunk):
    ctx = tess.tess_init(0)
    try:
        tess.tess_set_chunk_bytes(ctx, chunk)
        lo, hi = 100.0, 2500.0
        p = tess.process(8, precision=tess.TESS_FP32_DS, pt_min=pt_min, dr_min=0.4 if pt_min > 1 else 0.0,
                         eta_max=2.5 if pt_min > 1 else 50.0, hist_bins=bins, hist_observable=tess.TESS_OBS_HT,
                         hist_lo=lo, hist_hi=hi)
        tess.tess_select_variant(ctx, p, tess.TESS_K2_WAVE2U, tess.TESS_SCHED_SERIAL_HIST)
        assert tess.tess_plan_info(ctx, p, N)["schedule"] == tess.TESS_SCHED_SERIAL_HIST
        run = tess.Run(ctx, p, N)
        run.generate(2, 77)
        torch.cuda.synchronize()
        ok = run.t["pass"].cpu().numpy() != 0
        w, ht = run.t["weight"].cpu().numpy()[ok], run.t["ht"].cpu().numpy()[ok]
        b = 1 + np.floor((ht - lo) * (bins / (hi - lo))).astype(np.int64)
        b = np.where(ht < lo, 0, np.where(ht >= hi, bins + 1, np.minimum(b, bins)))
        hw, hw2 = (np.asarray(x) for x in run.histograms())
        for h, x in ((hw, w), (hw2, w * w)):
            ref = np.bincount(b, weights=x, minlength=bins + 2)
            # sums of up to N positive doubles in another order: N eps
            assert np.all(np.abs(h - ref) <= 1e-10 * ref), np.max(np.abs(h - ref))
    finally:
        tess.tess_destroy(ctx)
