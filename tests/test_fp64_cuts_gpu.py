"""The FP64 kinematics decide the pseudorapidity and Delta R cuts from FP32
estimates wherever those are clear of the cut: cut values next to an event's own
pseudorapidity or smallest Delta R, inside and outside the estimates' error,
against the oracle; and R_min of every event."""
import numpy as np
import pytest
import torch

import paper_1002_3446_gb300 as tess

pytestmark = pytest.mark.gpu


def _flags(ctx, n, first, N, **kw):
    run = tess.Run(ctx, tess.process(n, precision=tess.TESS_FP64, pt_min=1e-3, **kw), N)
    run.generate(7, first)
    torch.cuda.synchronize()
    return run.t["pass"].cpu().numpy(), run.t["rmin"].cpu().numpy()


# relative distance of the cut from the event's value: FP64 rounding of two
# implementations is below 1e-10, the estimates' error 2e-5 absolute
@pytest.mark.parametrize("n", [4, 5, 8, 12])
@pytest.mark.parametrize("off", [1e-9, 1e-6, 1e-4])
def test_cuts_next_to_an_events_own_values(n, off):
    import oracle as orc
    ctx = tess.tess_init(0)
    try:
        for ev in range(40, 52):
            r = orc.event(orc.process(n, pt_min=1e-3, eta_max=50.0, dr_min=0.0), 7, ev)
            if not r["pass"]:
                continue
            k = np.asarray(r["k"])[2:]
            eta = np.abs(np.arcsinh(k[:, 3] / np.hypot(k[:, 1], k[:, 2])) + r["y"])
            for side in (1 - off, 1 + off):
                ok, rmin = _flags(ctx, n, ev, 1, eta_max=float(eta.max() * side), dr_min=0.0)
                assert bool(ok[0]) == (side > 1), (ev, side)
                assert np.isclose(rmin[0], r["rmin"], rtol=1e-10)
                ok, _ = _flags(ctx, n, ev, 1, eta_max=50.0, dr_min=float(r["rmin"] / side))
                assert bool(ok[0]) == (side > 1), (ev, side)
    finally:
        tess.tess_destroy(ctx)


@pytest.mark.parametrize("n", [4, 6, 9, 12])
def test_rmin_of_many_events(n):
    import oracle as orc
    ctx = tess.tess_init(0)
    try:
        N = 20_001
        _, rmin = _flags(ctx, n, 0, N)
        ref = orc.generate(orc.process(n, pt_min=1e-3), 7, 0, N, hist=False)["rmin"]
        # the oracle's ln((|p| + pz) / (|p| - pz)) loses e^(2 |eta|) ulp, so its forward
        # pairs (|eta| up to about 8 in a sample of this size) set the tail
        rel = np.abs(rmin / ref - 1)
        assert np.median(rel) < 1e-14 and np.quantile(rel, 0.99) < 1e-11 and rel.max() < 1e-6
    finally:
        tess.tess_destroy(ctx)
