"""The blocks' rows of partial sums are written, not added to, by a call's first
chunk, so nothing in the workspace has to be cleared: sums and histograms from a
workspace full of NaN, in every epilogue (in the amplitude kernel, deferred, in
the one-kernel form, cut-first), one chunk and several, fewer tiles than blocks
and more."""
import numpy as np
import pytest
import torch

import paper_1002_3446_gb300 as tess

pytestmark = pytest.mark.gpu

FORMS = [(6, tess.TESS_HEL_SAMPLE, tess.TESS_K2_FUSED, 0, 0), (6, tess.TESS_HEL_SAMPLE, tess.TESS_K2_REG_HI, 0, 0),
         (6, tess.TESS_HEL_SAMPLE, tess.TESS_K2_REG_TMA, 4, 0), (10, tess.TESS_HEL_SAMPLE, tess.TESS_K2_WAVE2U, 4, 0),
         (8, tess.TESS_POL_RANDOM, tess.TESS_K2_REAL, 1, tess.TESS_FLAG_CUT_FIRST),
         (10, tess.TESS_POL_RANDOM, tess.TESS_K2_ROWS_REAL, 3, 0), (12, tess.TESS_HEL_SAMPLE, tess.TESS_K2_LANES16, 0, 0),
         (9, tess.TESS_HEL_SAMPLE, tess.TESS_K2_PAIR64, 0, 0), (9, tess.TESS_HEL_SAMPLE, tess.TESS_K2_WAVE2PU, 2, 0)]


@pytest.mark.parametrize("n,mode,form,sched,flags", FORMS)
@pytest.mark.parametrize("N,chunk", [(1, 0), (129, 0), (30_001, 1 << 20), (200_003, 0)])
def test_rows_need_no_clearing(n, mode, form, sched, flags, N, chunk):
    ctx = tess.tess_init(0)
    try:
        tess.tess_set_chunk_bytes(ctx, chunk)
        p = tess.process(n, precision=tess.TESS_FP32_DS, helicity_mode=mode, flags=flags, hist_bins=24,
                         hist_observable=tess.TESS_OBS_HT, hist_lo=100.0, hist_hi=2500.0)
        tess.tess_select_variant(ctx, p, form, sched)
        run = tess.Run(ctx, p, N)
        for _ in range(2):
            run.workspace.fill_(float("nan"))
            run.reset()
            run.generate(11, 5)
            torch.cuda.synchronize()
            w = run.t["weight"].cpu().numpy()
            acc = run.acc.cpu().numpy()
            # sums of N doubles in another order: N eps of the sum of magnitudes
            assert abs(acc[0] + acc[4] - w.sum()) <= 1e-12 * np.abs(w).sum()
            assert abs(acc[1] + acc[5] - (w * w).sum()) <= 1e-12 * (w * w).sum()
            assert acc[2] == run.t["pass"].cpu().numpy().sum() and acc[3] == N and acc[6] == 0 and acc[7] == 0
            hw, hw2 = run.histograms()
            assert abs(hw.sum() - w.sum()) <= 1e-12 * np.abs(w).sum()
            assert abs(hw2.sum() - (w * w).sum()) <= 1e-12 * (w * w).sum()
    finally:
        tess.tess_destroy(ctx)


@pytest.mark.parametrize("tiles", [1, 127, 1023, 1025, 9000])
def test_persistent_fold(tiles):
    """The persistent form's fold (a cluster of blocks per column): tile counts
    around its slices, two processes of different lengths."""
    ctx = tess.tess_init(0)
    try:
        procs = [tess.process(4, precision=tess.TESS_FP32_DS, hist_bins=10, hist_observable=tess.TESS_OBS_HT,
                              hist_lo=100.0, hist_hi=2500.0), tess.process(6, precision=tess.TESS_FP32_DS)]
        counts = [128 * tiles - 5, 128 * (tiles // 3) + 1]
        runs = [tess.Run(ctx, p, c) for p, c in zip(procs, counts)]
        ws = torch.full(((tess.tess_workspace_size_persistent(ctx, procs, counts) + 7) // 8,), float("nan"),
                        dtype=torch.float64, device="cuda")
        tess.tess_generate_persistent(ctx, procs, [3, 4], [0, 9], counts, [r.outputs for r in runs], ws)
        torch.cuda.synchronize()
        for r, c in zip(runs, counts):
            w, acc = r.t["weight"].cpu().numpy(), r.acc.cpu().numpy()
            assert abs(acc[0] + acc[4] - w.sum()) <= 1e-12 * np.abs(w).sum()
            assert abs(acc[1] + acc[5] - (w * w).sum()) <= 1e-12 * (w * w).sum()
            assert acc[2] == r.t["pass"].cpu().numpy().sum() and acc[3] == c
        hw, _ = runs[0].histograms()
        assert abs(hw.sum() - runs[0].t["weight"].sum().item()) <= 1e-12 * runs[0].t["weight"].abs().sum().item()
    finally:
        tess.tess_destroy(ctx)
