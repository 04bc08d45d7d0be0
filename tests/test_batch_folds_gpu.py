"""The folds of a batch in one launch, and one after another where processes share
accumulators: bit for bit the sums and histograms of separate calls in order."""
import pytest
import torch

import paper_1002_3446_gb300 as tess

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("share", [False, True])
@pytest.mark.parametrize("counts", [[5], [1, 127, 40_001], [300, 0, 129], [64] * 16])
def test_batch_folds(share, counts):
    ctx = tess.tess_init(0)
    try:
        k = len(counts)
        procs = [tess.process(4 + (0 if share else i % 3), precision=tess.TESS_FP32_DS,
                              hist_bins=0 if not share and i % 3 == 1 else 12, hist_observable=tess.TESS_OBS_HT,
                              hist_lo=100.0, hist_hi=2500.0) for i in range(k)]
        firsts, seeds = [1000 * i for i in range(k)], [3 + i for i in range(k)]
        ref = [tess.Run(ctx, p, max(c, 1)) for p, c in zip(procs, counts)]
        got = [tess.Run(ctx, p, max(c, 1)) for p, c in zip(procs, counts)]
        for runs in (ref, got):
            for r, c in zip(runs, counts):
                r.n_events = c
                if share:
                    r.acc, r.hist = runs[0].acc, runs[0].hist
                    r.outputs = tess.make_outputs(r.t["weight"], r.t["me2"], r.t["pass"], r.t["ht"], r.t["ptlead"],
                                                  r.t["rmin"], r.acc, r.hist)
        ws = torch.empty((tess.tess_workspace_size_batched(ctx, procs, counts) + 7) // 8, dtype=torch.float64,
                         device="cuda")
        for _ in range(2):  # capture, then replay into the same accumulators
            for r, s, f in zip(ref, seeds, firsts):
                r.generate(s, f)
            tess.tess_generate_batched(ctx, procs, seeds, firsts, counts, [r.outputs for r in got], ws)
        torch.cuda.synchronize()
        for a, b, c in zip(ref, got, counts):
            assert torch.equal(a.acc, b.acc) and a.acc[3] >= 2 * c
            assert a.hist is None or torch.equal(a.hist, b.hist)
    finally:
        tess.tess_destroy(ctx)
