"""The list of a cut-first chunk's passing events (scan of the tiles' counts in
rounds of lines per warp, then one warp per tile): counts around a tile, a line, a
warp's rounds and the block's, against a call that evaluates every event."""
import numpy as np
import pytest
import torch

import paper_1002_3446_gb300 as tess

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles,extra", [(0, 1), (1, -1), (31, 5), (32, 1), (512, -7), (512, 1), (16384, 0), (16384, 1),
                                         (33000, 77)])
@pytest.mark.parametrize("pt_min", [1.0, 20.0, 3000.0])
def test_list(tiles, extra, pt_min):
    N = 128 * tiles + extra
    ctx = tess.tess_init(0)
    try:
        got = []
        for flags in (tess.TESS_FLAG_CUT_FIRST, 0):
            p = tess.process(4, precision=tess.TESS_FP32_DS, pt_min=pt_min, flags=flags)
            tess.tess_select_variant(ctx, p, tess.TESS_K2_REG, 0)
            assert tess.tess_plan_info(ctx, p, N)["chunks"] == 1
            run = tess.Run(ctx, p, N, per_event=("weight", "pass"))
            run.generate(6, 11)
            torch.cuda.synchronize()
            got.append((run.t["weight"].cpu().numpy(), run.t["pass"].cpu().numpy(), run.acc.cpu().numpy()))
        (w, ok, acc), (w0, ok0, _) = got
        assert np.array_equal(ok, ok0) and np.all(w[ok == 0] == 0.0)
        # the same amplitude kernel on the same inputs
        assert np.array_equal(w, w0)
        assert acc[2] == ok.sum() and acc[3] == N and abs(acc[0] + acc[4] - w.sum()) <= 1e-12 * w.sum()
    finally:
        tess.tess_destroy(ctx)
