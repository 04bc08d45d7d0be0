"""The exact sum over helicities and colour orderings (n = 4, 5) event by event
against the oracle, which evaluates every ordering and labelling with
four-component currents: sizes around the tile of 128 events, every precision."""
import numpy as np
import pytest
import torch

import paper_1002_3446_gb300 as tess

pytestmark = pytest.mark.gpu

# FP64: rounding of two different recursions, 1e-10 as everywhere (single
# events near a collinear pole amplify it by 1 / s_min, see 16 x the oracle's
# own sensitivity below).  FP32: currents of a few dozen operations from
# momenta rounded once (6e-8), an invariant or two of which enters inverted;
# no labelling's suppression shows in the sum.
RTOL = {tess.TESS_FP64: 1e-10, tess.TESS_FP32_CURRENTS: 2e-4, tess.TESS_FP32_DS: 2e-4}


@pytest.mark.parametrize("n", [4, 5])
@pytest.mark.parametrize("precision", sorted(RTOL))
@pytest.mark.parametrize("N", [1, 127, 129, 300])
def test_exact_sum_events(n, precision, N):
    import oracle as orc
    ctx = tess.tess_init(0)
    try:
        p = tess.process(n, precision=precision, helicity_mode=tess.TESS_HEL_SUM)
        run = tess.Run(ctx, p, N)
        first = (1 << 33) + 7
        run.generate(3, first)
        torch.cuda.synchronize()
        me2, w = run.t["me2"].cpu().numpy(), run.t["weight"].cpu().numpy()
        op = orc.process(n, hel_mode=0)
        for i in range(N):
            r = orc.event(op, 3, first + i)
            rel = abs(me2[i] - r["me2"]) / r["me2"]
            if r["pass"]:
                rel = max(rel, abs(w[i] - r["weight"]) / r["weight"])
            assert rel <= RTOL[precision] or rel <= 16 * orc.ulp_sensitivity(op, 3, first + i), (i, rel)
    finally:
        tess.tess_destroy(ctx)
