"""The work that users of the generator have it do, as measurable cases.

A case is one call of a public entry point (or one short sequence of them, as
the autograd weight) at a stated size:

  api "generate"    tess_generate through ``Run``: reset, generate; per-event
                    arrays, the sums and the histogram come back
  api "batched"     tess_generate_batched over gg -> 2..10 gluons
  api "persistent"  tess_generate_persistent over the same kind of batch
  api "weights"     event_weight and its backward pass: a training step's
                    weights and gradients from given draws
  api "me2"         tess_me2: |A|^2 of momenta that the caller brings

``exact`` restates the whole path in plain float64 torch from its published
definitions (Philox4x32-10, Rambo, the Berends-Giele recursion with explicit
three- and four-gluon vertices); gradients are torch's own automatic
derivatives of that restatement.
"""
from __future__ import annotations

import itertools
import math

import torch

import paper_1002_3446_gb300 as tess

PRECISIONS = {"fp64": tess.TESS_FP64, "fp32": tess.TESS_FP32_CURRENTS, "ds": tess.TESS_FP32_DS}
MODES = {"sum": tess.TESS_HEL_SUM, "sample": tess.TESS_HEL_SAMPLE, "random": tess.TESS_POL_RANDOM}
OBSERVABLES = {"ptlead": tess.TESS_OBS_PTLEAD, "ht": tess.TESS_OBS_HT, "rmin": tess.TESS_OBS_RMIN}
HIST_RANGE = {"ptlead": (20.0, 1020.0), "ht": (200.0, 3000.0), "rmin": (0.0, 5.0)}
PER_EVENT = {"few": ("weight", "pass"), "obs": ("weight", "pass", "ht", "ptlead", "rmin"),
             "all": ("weight", "me2", "pass", "ht", "ptlead", "rmin")}

# api, n gluons, events, precision, helicity mode; then the options of a generation call: flags, cuts, histogram,
# which per-event arrays, whether they are pinned host memory, and whether the program tunes its context first.
# |A|^2 of events that fail the cuts has no use and no useful comparison (in single precision the norm of a sample is
# carried by its one event closest to a pole): "all" is asked for in double precision and with cut-first generation.
GENERATE = dict(api="generate", mode="sample", cut_first=False, pdf_grid=False, pt_min=20.0, eta_max=2.5, hist="",
                bins=0, out="few", host=False, tuned=False)


def listed():
    g = GENERATE
    return [
        # a handful of events with observables and a histogram: an interactive look or the step of an adaptive loop
        dict(g, name="gg2g small", n=4, events=1000, precision="ds", hist="ptlead", bins=50, out="obs"),
        # the flagship run: gg -> 4 gluons, 2^24 events, tuned once at start-up as the benchmark does
        dict(g, name="gg4g flagship", n=6, events=1 << 24, precision="ds", tuned=True),
        # a ragged chunk of a longer run on the second cut set (60 GeV, 2.0), native-FP64 boost, tabulated PDF
        dict(g, name="gg5g tabulated", n=7, events=500_009, precision="fp32", pdf_grid=True, pt_min=60.0, eta_max=2.0,
             hist="rmin", bins=50),
        # the README's example: gg -> 8 gluons, H_T histogram, per-event observables, built-in defaults
        dict(g, name="gg8g example", n=10, events=1 << 22, precision="ds", pt_min=30.0, hist="ht", bins=40, out="obs"),
        # the same physics as production runs it: tuned
        dict(g, name="gg8g tuned", n=10, events=1 << 22, precision="ds", pt_min=30.0, hist="ht", bins=40, tuned=True),
        # unweighting feed: random real polarisations, amplitudes for passing events only, results straight to the host
        dict(g, name="gg6g cut first", n=8, events=(1 << 21) + 77, precision="ds", mode="random", cut_first=True,
             out="all", host=True, tuned=True),
        # the plain FP64 form, as the accuracy reference of a production sample
        dict(g, name="gg4g double", n=6, events=1 << 20, precision="fp64", out="all"),
        # exact helicity and colour sum, FP64, leading-pT histogram
        dict(g, name="gg2g exact sum", n=4, events=1 << 20, precision="fp64", mode="sum", hist="ptlead", bins=50,
             out="all"),
        # every multiplicity of a jet-rate study in one call, as one graph
        dict(name="batch", api="batched", n=12, events=1 << 22, precision="ds", pt_min=20.0),
        # the same with one persistent launch
        dict(name="persistent batch", api="persistent", n=12, events=1 << 20, precision="ds", pt_min=20.0),
        # a training step through the event weight: weights, d/du and d/dln(mu_R)
        dict(name="gg6g weights", api="weights", n=8, events=1 << 18, precision="ds", pt_min=20.0),
        # matrix elements of an outside phase-space generator's events
        dict(name="gg6g matrix elements", api="me2", n=8, events=1 << 18, precision="fp64"),
    ]


def draw(rng):
    api = rng.choice(["generate"] * 6 + ["batched", "persistent", "weights", "me2"])
    n = rng.randint(4, 12)
    prec = rng.choice(["ds", "ds", "fp32", "fp64"])

    def events(case, low=1000):
        # from a size at which some events pass and are not zero by their helicities, log-uniform up to a size that costs less than the largest listed case, never above 2^23
        top = min(2e11 / _cost(case), 1 << (19 if case["api"] == "me2" else 23))
        return int(math.exp(rng.uniform(math.log(low), math.log(top))))

    if api == "generate":
        mode = rng.choice(["sample", "sample", "random"] + (["sum"] if n <= 5 else []))
        fast = prec != "fp64" and mode != "sum"
        hist = rng.choice(["", "ptlead", "ht", "rmin"])
        paper = rng.random() < 0.25
        case = dict(GENERATE, n=n, events=1, precision=prec, mode=mode, cut_first=fast and rng.random() < 0.3,
                    pdf_grid=fast and rng.random() < 0.2, pt_min=60.0 if paper else rng.choice([20.0, 30.0]),
                    eta_max=2.0 if paper else 2.5, hist=hist, bins=rng.choice([1, 40, 50, 200]) if hist else 0,
                    out="few", host=rng.random() < 0.2, tuned=mode != "sum" and rng.random() < 0.4)
        case["out"] = rng.choice(["few", "obs"] + (["all"] if prec == "fp64" or case["cut_first"] else []))
    elif api in ("batched", "persistent"):
        case = dict(api=api, n=rng.randint(5, 12), events=1, precision="ds" if api == "persistent" else prec, pt_min=20.0)
    elif api == "weights":
        case = dict(api=api, n=n, events=1, precision=prec, pt_min=rng.choice([20.0, 30.0]))
    else:
        case = dict(api=api, n=n, events=1, precision=prec)
    case["events"] = events(case, low=1 << 14 if api in ("batched", "persistent") else 1000)
    return case


# --------------------------------------------------------------------------- work
def _amplitude_flops(n):
    """One colour-ordered amplitude: each current has two physical (transverse) complex components, so a split needs
    one complex product of two such vectors, two with momenta and two scalings (84 operations), a four-gluon triple one
    product and one scaling (30), and a current its propagator (40)."""
    legs = n - 1
    return 84 * math.comb(legs + 1, 3) + 30 * math.comb(legs + 1, 4) + 40 * legs * (legs - 1) // 2


def _flops(case, n):
    amps, m = 1.0, n - 2
    if case.get("mode") == "random":
        amps = 0.25  # real currents: a quarter of the multiplications
    elif case.get("mode") == "sum":
        amps = math.factorial(n - 1) / 2 * (2 ** (n - 1) - 1 - n)  # orderings and labellings that are not equal or zero
    if case.get("cut_first"):
        amps *= 0.1  # about the share of events that passes
    if case["api"] == "me2":
        return amps * _amplitude_flops(n) + 20 * n
    if case["api"] == "weights":  # forward, and about three times that for the reverse sweep
        return 4 * _amplitude_flops(n) + 400 * m
    # draws (ten rounds of Philox per two uniforms), seeds, boost, cuts, pairwise distances
    return amps * _amplitude_flops(n) + 250 * m + 6 * m * (m - 1)


def _cost(case):
    """Rough operations per event (of the smallest n, in a batch), FP64 ones counted at their rate on this GPU."""
    case = dict(case, cut_first=False, mode="sum" if case.get("mode") == "sum" else "sample")
    c = _flops(case, case["n"]) * 2
    if case["api"] in ("batched", "persistent"):
        c = sum(_flops(case, n) / 2 ** (n - 4) for n in range(4, case["n"] + 1)) * 2
    if case["mode"] == "sum":
        c *= 4
    if case["precision"] == "fp64":
        c *= 40
    return c * (8 if case["api"] == "weights" else 1)


def _members(case):
    """(n, events) of a batch: 4..n gluons, events halving with each further gluon."""
    return [(n, max(1, case["events"] >> (n - 4))) for n in range(4, case["n"] + 1)]


def work(case):
    if case["api"] in ("batched", "persistent"):
        return {"bytes": float(sum(9 * e for _, e in _members(case))),
                "flops": float(sum(e * _flops(case, n) for n, e in _members(case)))}
    n, e = case["n"], case["events"]
    if case["api"] == "generate":
        per = {"few": 9, "obs": 33, "all": 41}[case["out"]]
    elif case["api"] == "me2":
        per = 32 * n + n + 4 + 8
    else:  # draws, labels and ordering in, upstream gradient in; weight and gradients out
        nu = 2 + 4 * (n - 2)
        per = 8 * nu + 4 + n + 8 + 8 + 8 * nu
    return {"bytes": float(per * e), "flops": float(e * _flops(case, n))}


def tolerance(case):
    # FP64: every step in double.  Weights and |A|^2 span many decades and their norms are carried by the events next
    # to collinear poles, which amplify rounding by the inverse of the smallest invariant (seen against float64 torch:
    # up to 5e-12 of the norm, 3e-10 in one event).
    if case["precision"] == "fp64":
        return {"rel": 2e-11 if case["api"] != "weights" else 1e-10, "max": 1e-8, "differ": 4e-6}
    # FP32 currents: the same amplification of 6e-8 (seen: up to 4.4e-4 of the norm, 0.9 in one strongly boosted event;
    # 2e-7 of the cut decisions, which the FP32 forms take on rounded momenta).
    return {"rel": 2e-3, "max": 0.99, "differ": 4e-6}


# --------------------------------------------------------------------------- the program
_contexts = {}


def _context(case):
    """A program keeps its context; one that tunes it keeps a context per kind of run."""
    key = None
    if case.get("tuned"):
        key = tuple(case[k] for k in ("n", "events", "precision", "mode", "cut_first", "pdf_grid", "bins", "out", "host"))
    new = key not in _contexts
    if new:
        _contexts[key] = tess.tess_init(torch.cuda.current_device())
    return _contexts[key], new


def _process(case, n=None):
    kw = {}
    if case.get("bins"):
        lo, hi = HIST_RANGE[case["hist"]]
        kw = dict(hist_observable=OBSERVABLES[case["hist"]], hist_bins=case["bins"], hist_lo=lo, hist_hi=hi)
    flags = (tess.TESS_FLAG_CUT_FIRST if case.get("cut_first") else 0) | (
        tess.TESS_FLAG_PDF_GRID if case.get("pdf_grid") else 0)
    return tess.process(n or case["n"], precision=PRECISIONS[case["precision"]],
                        helicity_mode=MODES[case.get("mode", "sample")], pt_min=case.get("pt_min", 20.0),
                        eta_max=case.get("eta_max", 2.5), flags=flags, **kw)


def prepare(case, seed):
    ctx, new = _context(case)
    api, n, events = case["api"], case["n"], case["events"]
    if api == "generate":
        proc = _process(case)
        run = tess.Run(ctx, proc, events, per_event=PER_EVENT[case["out"]], host_per_event=case["host"])
        if new and case["tuned"]:
            tess.tess_autotune(ctx, proc, min(events, 1 << 22), None, run.workspace, outputs=run.outputs)
        return dict(case=case, run=run, seed=seed, first=_first(seed))
    if api in ("batched", "persistent"):
        members = _members(case)
        procs = [_process(case, m) for m, _ in members]
        counts = [e for _, e in members]
        outs = [dict(weight=torch.empty(e, dtype=torch.float64, device="cuda"),
                     pass_=torch.empty(e, dtype=torch.uint8, device="cuda")) for e in counts]
        acc = torch.zeros((len(members), tess.TESS_ACC_LEN), dtype=torch.float64, device="cuda")
        size = tess.tess_workspace_size_batched if api == "batched" else tess.tess_workspace_size_persistent
        ws = torch.empty((size(ctx, procs, counts) + 7) // 8, dtype=torch.float64, device="cuda")
        return dict(case=case, ctx=ctx, procs=procs, counts=counts, outs=outs, acc=acc, workspace=ws,
                    seeds=[seed + m for m, _ in members], first=[_first(seed)] * len(members),
                    outputs=[tess.make_outputs(acc=a, **o) for a, o in zip(acc, outs)])
    if api == "weights":
        u, hel, order = tess.tess_draws(ctx, n, seed, _first(seed), events)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        up = torch.rand(events, generator=gen, dtype=torch.float64, device="cuda") + 0.5
        return dict(case=case, ctx=ctx, proc=_process(case), u=u, hel=hel, order=order, up=up)
    k, order, hel = _outside_events(n, events, seed)
    return dict(case=case, ctx=ctx, k=k, order=order, hel=hel,
                me2=torch.empty(events, dtype=torch.float64, device="cuda"))


def _first(seed):
    """Where in its stream a run starts: a resumed run does not start at event 0."""
    return (seed % 1009) * 4099


def run(state):
    case = state["case"]
    if case["api"] == "generate":
        r = state["run"]
        r.reset()
        r.generate(state["seed"], state["first"])
        out = {k: t for k, t in r.t.items() if t is not None}
        return _with_sums(out, r.acc, r.hist, case["bins"])
    if case["api"] in ("batched", "persistent"):
        state["acc"].zero_()
        call = tess.tess_generate_batched if case["api"] == "batched" else tess.tess_generate_persistent
        call(state["ctx"], state["procs"], state["seeds"], state["first"], state["counts"], state["outputs"],
             state["workspace"])
        return [_with_sums({"weight": o["weight"], "pass": o["pass_"]}, a, None, 0)
                for o, a in zip(state["outs"], state["acc"])]
    if case["api"] == "weights":
        u = state["u"].detach().requires_grad_(True)
        log_xi = torch.zeros((), dtype=torch.float64, device="cuda", requires_grad=True)
        w = tess.event_weight(state["ctx"], state["proc"], u, state["hel"], state["order"], log_xi)
        gu, gxi = torch.autograd.grad(w, [u, log_xi], state["up"])
        return {"w": w.detach(), "grad_u": gu, "grad_log_xi": gxi}
    tess.tess_me2(state["ctx"], case["n"], PRECISIONS[case["precision"]], state["k"], state["order"], state["hel"],
                  state["me2"])
    return {"me2": state["me2"]}


def _with_sums(out, acc, hist, bins):
    """Per-event arrays and the sums; the sums' compensation terms (rounding residues) are left to the next call."""
    out.update(sum_w=acc[0:1], sum_w2=acc[1:2], counts=acc[2:4], faults=acc[6:8])
    if bins:
        out.update(hist_w=hist[: bins + 2], hist_w2=hist[bins + 2: 2 * (bins + 2)])
    return out


# --------------------------------------------------------------------------- the same path in float64
F64 = dict(dtype=torch.float64, device="cuda")
M32 = 0xFFFFFFFF


def _mul32(c, x):
    """High and low words of the 64-bit product of a constant and 32-bit words held in int64."""
    t = c * (x & 0xFFFF)
    s = c * (x >> 16) + (t >> 16)
    return s >> 16, ((s & 0xFFFF) << 16) | (t & 0xFFFF)


def _philox(seed, ev, blk):
    c = [ev & M32, (ev >> 32) & M32, torch.full_like(ev, blk), torch.zeros_like(ev)]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        h0, l0 = _mul32(0xD2511F53, c[0])
        h1, l1 = _mul32(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


class _Draws:
    """Uniform j of each event, and the words behind it."""

    def __init__(self, seed, ev):
        self.seed, self.ev, self.blocks = seed, ev, {}

    def words(self, j):
        if j >> 1 not in self.blocks:
            self.blocks[j >> 1] = _philox(self.seed, self.ev, j >> 1)
        w = self.blocks[j >> 1]
        return (w[2], w[3]) if j & 1 else (w[0], w[1])

    def u(self, j):
        a, b = self.words(j)
        return (((a >> 6) << 26) | (b >> 6)).double() * 2.0**-52 + 2.0**-53


def _configuration(n, d):
    """Helicity bits and colour ordering of each event."""
    j = 2 + 4 * (n - 2)
    hel = d.words(j)[0] >> (32 - n)
    order = torch.arange(n, device="cuda").repeat(d.ev.numel(), 1)
    for i in range(n, 2, -1):
        r = 1 + torch.floor(d.u(j + 1 + n - i) * (i - 1)).long()  # position (from 0) that position i - 1 changes with
        here, there = order[:, i - 1].clone(), order.gather(1, r[:, None])
        order.scatter_(1, r[:, None], here[:, None])
        order[:, i - 1] = there[:, 0]
        same = r == i - 1
        order[same, i - 1] = here[same]
    return hel, order


def _phase_space(n, u, lnxmin, s_had):
    """Rambo momenta k[leg][4] (all outgoing), x1, x2, s_hat from the uniforms u[j]."""
    m = n - 2
    x = [torch.exp(u[0] * lnxmin), torch.exp(u[1] * lnxmin)]
    shat = x[0] * x[1] * s_had
    rs = torch.sqrt(shat)
    q = []
    for i in range(m):
        c = 2 * u[2 + 4 * i] - 1
        s = torch.sqrt(1 - c * c)
        phi = 2 * math.pi * u[3 + 4 * i]
        e = -torch.log(u[4 + 4 * i] * u[5 + 4 * i])
        q.append([e, e * s * torch.cos(phi), e * s * torch.sin(phi), e * c])
    tot = [sum(p[j] for p in q) for j in range(4)]
    mass = torch.sqrt(tot[0] ** 2 - tot[1] ** 2 - tot[2] ** 2 - tot[3] ** 2)
    b = [-tot[j] / mass for j in (1, 2, 3)]
    gam = tot[0] / mass
    a, scale = 1 / (1 + gam), rs / mass
    zero = torch.zeros_like(rs)
    k = [[-rs / 2, zero, zero, -rs / 2], [-rs / 2, zero, zero, rs / 2]]
    for p in q:
        bq = b[0] * p[1] + b[1] * p[2] + b[2] * p[3]
        f = a * bq + p[0]
        k.append([scale * (gam * p[0] + bq)] + [scale * (p[1 + j] + b[j] * f) for j in range(3)])
    return k, x, shat


def _observables(case, k, x):
    y = 0.5 * torch.log(x[0] / x[1])
    ok = torch.ones_like(y, dtype=torch.bool)
    pt, eta, phi = [], [], []
    for _, px, py, pz in k[2:]:
        t = torch.sqrt(px * px + py * py)
        pt.append(t)
        eta.append(torch.asinh(pz / t) + y)
        phi.append((px, py))
        ok &= (t > case.get("pt_min", 20.0)) & (eta[-1].abs() < case.get("eta_max", 2.5))
    r2 = torch.full_like(y, math.inf)
    for i, j in itertools.combinations(range(len(pt)), 2):
        (xi, yi), (xj, yj) = phi[i], phi[j]
        dphi = torch.atan2((xi * yj - yi * xj).abs(), xi * xj + yi * yj)
        d = (eta[i] - eta[j]) ** 2 + dphi**2
        r2 = torch.minimum(r2, d)
        ok &= d > 0.4**2
    return ok, sum(pt), torch.stack(pt).amax(0), torch.sqrt(r2)


def _polarisation(leg, k, label=None, angle=None):
    """(4, events) polarisation vectors of physical momenta: by helicity label (0: eps_+), or a real vector by angle."""
    sg = -1.0 if leg < 2 else 1.0
    px, py, pz = (sg * k[j] for j in (1, 2, 3))
    pt2 = px * px + py * py
    axis = pt2 == 0
    pt = torch.sqrt(torch.where(axis, torch.ones_like(pt2), pt2))
    r = torch.sqrt(pt2 + pz * pz)
    ct, st = pz / r, torch.where(axis, torch.zeros_like(pt), pt) / r
    cf, sf = torch.where(axis, torch.ones_like(pt), px / pt), torch.where(axis, torch.zeros_like(pt), py / pt)
    zero = torch.zeros_like(ct)
    e1, e2 = torch.stack([zero, ct * cf, ct * sf, -st]), torch.stack([zero, -sf, cf, zero])
    if angle is not None:
        return torch.complex(torch.cos(angle) * e1 + torch.sin(angle) * e2, torch.zeros_like(e1))
    sign = torch.where(label.bool(), 1.0, -1.0).double()
    return torch.complex(sign * e1, -e2) / math.sqrt(2.0)


_metric = torch.tensor([1.0, -1.0, -1.0, -1.0], dtype=torch.float64)[:, None]


def _dot(a, b):
    return (a * b * _metric.to(a.device)).sum(0)


def _amplitude(k, eps):
    """m = eps[0] . K^2 J of the other legs; k, eps: lists over colour positions of (4, events)."""
    legs = len(k) - 1
    J, K = {}, {}
    for a in range(legs):
        J[a, a], K[a, a] = eps[a + 1], k[a + 1]
    for ln in range(2, legs + 1):
        for a in range(legs - ln + 1):
            b = a + ln - 1
            K[a, b] = K[a, b - 1] + K[b, b]
            num = 0
            for i in range(a, b):
                l, r = J[a, i], J[i + 1, b]
                kl, kr = K[a, i], K[i + 1, b]
                num = num + 2 * _dot(l, kr) * r - 2 * _dot(r, kl) * l + _dot(l, r) * (kl - kr)
            for i in range(a, b - 1):
                for j in range(i + 1, b):
                    A, B, C = J[a, i], J[i + 1, j], J[j + 1, b]
                    num = num + 2 * _dot(A, C) * B - _dot(A, B) * C - _dot(B, C) * A
            if ln == legs:
                return _dot(eps[0], num)
            J[a, b] = num / _dot(K[a, b], K[a, b])
    raise AssertionError


def _ordered(n, k, order, pol):
    """Momenta and polarisation vectors in colour order."""
    kk, ee = torch.stack([torch.stack(p) for p in k]), torch.stack(pol)  # [leg, 4, event]
    at = order.t()[:, None, :].expand(n, 4, -1)
    return list(kk.gather(0, at).unbind(0)), list(ee.gather(0, at).unbind(0))


def _amp2(n, k, hel=None, order=None, angles=None):
    pol = [_polarisation(l, k[l], None if hel is None else (hel >> l) & 1, None if angles is None else angles[l])
           for l in range(n)]
    kk, ee = _ordered(n, k, order, pol)
    return _amplitude(kk, ee).abs() ** 2


def _summed(n, k):
    """Sum of |m|^2 over 2^n helicities and (n-1)! orderings: flipping every label, and reversing the ordering, leave
    |m| as it is."""
    total = 0
    pols = [[_polarisation(l, k[l], torch.full_like(k[l][0], b)) for b in (0, 1)] for l in range(n)]
    kk = [torch.stack(p) for p in k]
    for perm in itertools.permutations(range(1, n)):
        if perm[0] > perm[-1]:
            continue
        order = (0,) + perm
        for hel in range(0, 2**n, 2):
            total = total + 4 * _amplitude([kk[l] for l in order], [pols[l][hel >> l & 1] for l in order]).abs() ** 2
    return total


def _table(x, nodes, values):
    """Linear interpolation between equidistant nodes at x in node units."""
    i = torch.clamp(x.long(), 0, nodes - 2)
    t = torch.clamp(x, 0, nodes - 1) - i
    return values[i] + t * (values[i + 1] - values[i])


def _weight_factor(case, n, u, x, shat, ht, mu_factor=0.5):
    """Weight over E: coupling, luminosity, flux, phase space."""
    m, s_had = n - 2, 14000.0**2
    lnxmin = math.log((m * case.get("pt_min", 20.0)) ** 2 / s_had)
    b0 = (33 - 10) / (12 * math.pi)

    def alphas(lnmu2):
        return 0.118 / (1 + 0.118 * b0 * (lnmu2 - math.log(91.19**2)))

    def density(z):
        return 1.7 * z**-0.2 * (1 - z) ** 5

    lnmu2 = 2 * torch.log(mu_factor * ht)
    if case.get("pdf_grid"):
        g = density(torch.exp(torch.arange(1025, **F64) / 1024 * lnxmin)).float().double()
        lum = _table(u[0] * 1024, 1025, g) * _table(u[1] * 1024, 1025, g)
        lo, hi = 2 * math.log(0.5 * m * case["pt_min"]), 2 * math.log(0.5 * 14000.0)
        a = alphas(lo + (hi - lo) * torch.arange(513, **F64) / 512).float().double()
        als = _table((lnmu2 - lo) / (hi - lo) * 512, 513, a)
    else:
        lum, als = density(x[0]) * density(x[1]), alphas(lnmu2)
    phase = (2 * math.pi) ** (4 - 3 * m) * (math.pi / 2) ** (m - 1) / (math.factorial(m - 1) * math.factorial(m - 2))
    const = 3.0 ** (n - 2) * 8 / (256 * math.factorial(m)) * 0.3893793721e9 * lnxmin**2 * phase / 2
    return const * lum * shat ** (m - 3) * (4 * math.pi * als) ** (n - 2)


def _generate_chunk(case, n, seed, first, count):
    d = _Draws(seed, torch.arange(first, first + count, device="cuda"))
    m, s_had = n - 2, 14000.0**2
    lnxmin = math.log((m * case["pt_min"]) ** 2 / s_had)
    u = [d.u(j) for j in range(2 + 4 * m)]
    k, x, shat = _phase_space(n, u, lnxmin, s_had)
    ok, ht, lead, rmin = _observables(case, k, x)
    mode = case.get("mode", "sample")
    if mode == "sum":
        e = _summed(n, k) / 2 ** (n - 2)
    else:
        hel, order = _configuration(n, d)
        angles = None
        if mode == "random":
            j0 = 2 + 4 * m + 1 + m
            angles, hel = [2 * math.pi * d.u(j0 + l) for l in range(n)], None
        e = _amp2(n, k, hel, order, angles) * 4 * math.factorial(n - 1)
    w = torch.where(ok, _weight_factor(case, n, u, x, shat, ht) * e, 0.0)
    if case.get("cut_first"):
        e = torch.where(ok, e, 0.0)
    return dict(weight=w, me2=e, ht=ht, ptlead=lead, rmin=rmin, ok=ok)


def _generate(case, n, seed, first, count, names):
    step = 1 << 17
    parts = [_generate_chunk(case, n, seed, first + i, min(step, count - i)) for i in range(0, count, step)]
    r = {k: torch.cat([p[k] for p in parts]) for k in parts[0]}
    w, ok = r["weight"], r["ok"]
    out = {k: ok.to(torch.uint8) if k == "pass" else r[k] for k in names}
    out.update(sum_w=w.sum()[None], sum_w2=(w * w).sum()[None],
               counts=torch.stack([ok.sum().double(), torch.tensor(float(count), **F64)]), faults=torch.zeros(2, **F64))
    if case.get("bins"):
        lo, hi = HIST_RANGE[case["hist"]]
        at = 1 + torch.floor((r[case["hist"]] - lo) * (case["bins"] / (hi - lo))).clamp(-1, case["bins"]).long()
        for key, v in (("hist_w", w), ("hist_w2", w * w)):
            out[key] = torch.zeros(case["bins"] + 2, **F64).index_add_(0, at[ok], v[ok])
    return out


def _outside_events(n, events, seed):
    """Momenta, colour orderings and helicity labels that a caller's own generator would bring: events within its cuts."""
    lnxmin = math.log(((n - 2) * 20.0) ** 2 / 14000.0**2)
    parts, have, first = [], 0, _first(seed)
    while have < events:
        d = _Draws(seed, torch.arange(first, first + (1 << 20), device="cuda"))
        k, x, _ = _phase_space(n, [d.u(j) for j in range(2 + 4 * (n - 2))], lnxmin, 14000.0**2)
        ok = _observables({}, k, x)[0]
        d = _Draws(seed, d.ev[ok])
        hel, order = _configuration(n, d)
        parts.append((torch.stack([torch.stack(p, -1) for p in k], 1)[ok], order.to(torch.uint8), hel.to(torch.int32)))
        have, first = have + hel.numel(), first + (1 << 20)
    return tuple(torch.cat(p)[:events].contiguous() for p in zip(*parts))


def _exact_weights(case, seed):
    n, count, step = case["n"], case["events"], 1 << 14
    gen = torch.Generator(device="cuda").manual_seed(seed)
    up = torch.rand(count, generator=gen, dtype=torch.float64, device="cuda") + 0.5
    lnxmin = math.log(((n - 2) * case["pt_min"]) ** 2 / 14000.0**2)
    ws, gs, gx = [], [], torch.zeros((), **F64)
    for i in range(0, count, step):
        c = min(step, count - i)
        d = _Draws(seed, torch.arange(_first(seed) + i, _first(seed) + i + c, device="cuda"))
        hel, order = _configuration(n, d)
        u = torch.stack([d.u(j) for j in range(2 + 4 * (n - 2))], 1).requires_grad_(True)
        log_xi = torch.zeros((), **F64).requires_grad_(True)
        cols = list(u.unbind(1))
        k, x, shat = _phase_space(n, cols, lnxmin, 14000.0**2)
        ok, ht, _, _ = _observables(case, [[v.detach() for v in p] for p in k], [v.detach() for v in x])
        ht = sum(torch.sqrt(p[1] ** 2 + p[2] ** 2) for p in k[2:])
        e = _amp2(n, k, hel, order) * 4 * math.factorial(n - 1)
        w = _weight_factor(case, n, cols, x, shat, ht, 0.5 * torch.exp(log_xi)) * e * ok
        a, b = torch.autograd.grad(w, [u, log_xi], up[i: i + c])
        ws.append(w.detach())
        gs.append(a)
        gx = gx + b
    return {"w": torch.cat(ws), "grad_u": torch.cat(gs), "grad_log_xi": gx}


def exact(case, seed):
    api, n = case["api"], case["n"]
    if api == "generate":
        return _generate(case, n, seed, _first(seed), case["events"], PER_EVENT[case["out"]])
    if api in ("batched", "persistent"):
        return [_generate(case, m, seed + m, _first(seed), e, PER_EVENT["few"]) for m, e in _members(case)]
    if api == "weights":
        return _exact_weights(case, seed)
    k, order, hel = _outside_events(n, case["events"], seed)
    out = []
    for i in range(0, case["events"], 1 << 17):
        s = slice(i, i + (1 << 17))
        legs = [list(p.unbind(1)) for p in k[s].unbind(1)]
        out.append(_amp2(n, legs, hel[s].long(), order[s].long()) / 2 ** (n - 2))
    return {"me2": torch.cat(out)}
