"""The calls that a program of this library spends its time in, with their inputs.

A multicanonical study iterates the weights (sweeps of many walkers, histogram
merge, weight update), then runs recorded production sweeps at fixed weights,
and then analyses the recorded series: reweighting to a grid of fields
Delta, the pseudo-transition point Delta*_L, the equal-height field.  Every
part is here at the sizes of the repository's own workloads
(``paper_1502_07214_gb300/workloads.py``), of the paper (L = 8 .. 28) and in
between:

  listed()        the named cases
  draw(rng)       one more case of the same ranges
  prepare(c, s)   what a program holds before the call (contexts with relaxed
                  walkers and weights, recorded series on the GPU)
  run(state)      one pass through the public entry points, outputs whole
  work(c)         bytes and operations that a pass cannot do without
  exact(c, s)     the same outputs in 64-bit torch arithmetic, for the analysis
                  calls (the simulation's outputs are integers, or weights that
                  have no value without running the whole chain)
"""
from fractions import Fraction

import numpy as np
import torch

from paper_1502_07214_gb300 import muca
from paper_1502_07214_gb300 import workloads as wl

# fields of the transition at the paper's temperatures (the bulk estimates of
# its Sec. IV and V), which give the slope of converged weights
FIELDS = {2.0: 2.523, 1.4182: 2.8446, 1.0: 2.944, 0.9: 2.964}
FIELD_T = 1.4182          # temperature of the synthetic series
FIELD_CENTRE = 2.8446     # and its transition field
# the benchmark's count of integer operations per update attempt
OPS_PER_ATTEMPT = 40


def listed():
    return [
        # the smallest run of the repository: 64 walkers of L = 8, where the
        # length of one walker's chain and the launches count
        dict(name="iterate_small", kind="iterate", L=8, T=2.0, walkers=64, sweeps=200),
        # an ordinary weight iteration near a first-order transition
        dict(name="iterate_medium", kind="iterate", L=16, T=1.0, walkers=1024, sweeps=500),
        # a weight iteration of a large lattice
        dict(name="iterate_large", kind="iterate", L=32, T=0.9, walkers=2048, sweeps=150),
        # many (L, T) groups in one context: the batched finite-size study
        dict(name="iterate_batch", kind="batch", walkers=512, sweeps=60),
        # a lattice whose rows are no multiple of four sites (the paper's sizes
        # are even numbers up to 28)
        dict(name="iterate_ragged", kind="iterate", L=22, T=1.4182, walkers=1000, sweeps=50),
        # recorded production sweeps at fixed weights, walkers spread over both
        # phases, at the paper's largest size
        dict(name="production_L28", kind="production", L=28, T=1.0, walkers=1024, sweeps=100),
        # the same at the benchmark's size: L = 48, 4096 walkers
        dict(name="production_L48", kind="production", L=48, T=0.9, walkers=4096, sweeps=60),
        # the disordered model: couplings per bond, one realisation
        dict(name="disordered_L24", kind="disordered", L=24, T=3.6, walkers=4096, sweeps=50),
        # a short series to a few fields, in 64 bits: launches and copies count
        dict(name="reweight_short", kind="reweight", L=12, walkers=64, samples=2000, grid=64,
             precision=64),
        # the whole series of a production run to a fine grid of fields
        dict(name="reweight_full64", kind="reweight", L=32, walkers=4096, samples=10000,
             grid=4096, precision=64),
        dict(name="reweight_full32", kind="reweight", L=32, walkers=4096, samples=10000,
             grid=4096, precision=32),
        # the pseudo-transition point and the equal-height field of the same
        # series, with jackknife errors
        dict(name="transition_L32", kind="transition", L=32, walkers=4096, samples=10000,
             blocks=20),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["iterate", "iterate", "iterate", "production", "production", "batch",
                       "disordered", "reweight", "reweight", "transition"])
    if kind in ("reweight", "transition"):
        L = rng.randint(8, 32)
        walkers = _log_int(rng, 32, 4096)
        samples = max(200000 // walkers + 1, _log_int(rng, 200, 10000))
        if kind == "transition":
            return dict(kind=kind, L=L, walkers=walkers, samples=samples,
                        blocks=rng.randint(2, 40))
        return dict(kind=kind, L=L, walkers=walkers, samples=samples,
                    grid=_log_int(rng, 16, 4096), precision=rng.choice([64, 32]))
    if kind == "batch":
        return dict(kind=kind, walkers=_log_int(rng, 64, 512), sweeps=rng.randint(20, 60))
    T = rng.choice(list(wl.TEMPS))
    L = rng.randint(4, 32) if rng.random() < 0.8 else 4 * rng.randint(8, 12)
    walkers = _log_int(rng, 32, 4096)
    if L > 32:
        walkers = min(walkers, 2048)
    if kind == "disordered":
        L = min(L, 28)
        T *= 4.0  # the couplings' mean is 4
    if kind == "production":
        walkers = max(32, min(walkers, 30_000_000 // L ** 3))
    # a pass of the size of the listed ones: bounded by the attempts of all
    # walkers and by one walker's sites
    slow = 5 if (L % 4 or kind == "disordered") else 1
    sweeps = min(500, int(2.0e10 / slow / (walkers * L ** 3)), int(3e6 / slow / L ** 3))
    return dict(kind=kind, L=L, T=T, walkers=walkers, sweeps=max(4, sweeps))


# ------------------------------------------------------------------ inputs
def _series(L, walkers, samples, seed):
    """A multicanonical series shaped like ``workloads.synthetic_series``, drawn
    on the GPU: E_Delta of every walker a random walk over [0, V], E_J and M
    around means that depend on it, weights whose reweighted distribution has
    two equal peaks at the transition field."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    V, beta = L ** 3, 1.0 / FIELD_T
    e = np.arange(V + 1, dtype=np.float64) / V
    well = -((e - 0.25) * (e - 0.8)) ** 2 / 0.01
    lnW = -(beta * FIELD_CENTRE * V * e + (0.6 * L * L) * (well - well.max()))
    step = max(1, V // 200)
    x0 = torch.randint(0, V + 1, (1, walkers), generator=g, device="cuda")
    dx = torch.randint(-step, step + 1, (samples, walkers), generator=g, device="cuda")
    x = (x0 + dx.cumsum(0)).remainder_(2 * V)
    ed = torch.where(x > V, 2 * V - x, x)
    del x, dx
    ef = ed.to(torch.float32) / V
    ej = -3.0 * V * ef ** 2 * (0.4 + 0.6 * ef)
    ej += V ** 0.5 * torch.randn(ef.shape, generator=g, device="cuda")
    sign = torch.where(torch.rand(walkers, generator=g, device="cuda") < 0.5, -1.0, 1.0)
    mag = V * ef * ((ef - 0.4) / 0.4).clamp_(0.0, 1.0)
    mag += V ** 0.5 * torch.randn(ef.shape, generator=g, device="cuda")
    m = torch.round(mag * sign).to(torch.int32)
    ed = ed.to(torch.int32)
    m = torch.minimum(torch.maximum(m, -ed), ed)
    return torch.round(ej).to(torch.int32), ed.contiguous(), m.contiguous(), lnW


def _half_width(L):
    """Half the width of a grid of fields around the transition: +-0.05 at
    L = 32, wider for smaller lattices (the transition rounds like 1 / V)."""
    return 0.05 * (32.0 / L) ** 1.5


def _spins(L, T, walkers, seed):
    """Walkers spread over the whole range of E_Delta near a transition: a slab
    of one of the two +-1 phases of random thickness in the vacancy phase, each
    with a few per cent of other spins."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    x = torch.arange(L ** 3, device="cuda") // (L * L)
    cut = torch.rand((walkers, 1), generator=g, device="cuda") * (L + 1)
    sign = torch.randint(0, 2, (walkers, 1), generator=g, device="cuda") * 2 - 1
    s = torch.where(x[None, :] < cut, sign, torch.zeros_like(sign)).to(torch.int8)
    hot = torch.rand(s.shape, generator=g, device="cuda") < (0.03 if T <= 1.0 else 0.3)
    other = torch.randint(-1, 2, s.shape, generator=g, device="cuda", dtype=torch.int8)
    return torch.where(hot, other, s).cpu().numpy()


def prepare(case, seed):
    kind, seed = case["kind"], int(seed)
    st = {"case": case}
    if kind in ("reweight", "transition"):
        L = case["L"]
        ej, ed, m, lnW = _series(L, case["walkers"], case["samples"], seed)
        beta, V, h = 1.0 / FIELD_T, L ** 3, _half_width(L)
        st.update(ej=ej, ed=ed, m=m, lnW=lnW, beta=beta, V=V)
        if kind == "reweight":
            st["grid"] = wl.delta_grid(FIELD_CENTRE, h, case["grid"])
        else:
            # the bracket of Delta*_L from a coarse scan of the same series
            coarse = wl.delta_grid(FIELD_CENTRE, h, 201)
            c = muca.reweight(ej, ed, m, lnW, 0, beta, V, coarse, 64)[:, 2]
            k = int(np.argmax(c))
            st.update(lo=float(coarse[max(k - 4, 0)]), hi=float(coarse[min(k + 4, 200)]),
                      split=int(0.525 * V), eq_lo=FIELD_CENTRE - h, eq_hi=FIELD_CENTRE + h)
        return st
    if kind == "batch":
        groups = wl.mixed_groups(n_walkers=case["walkers"])
    else:
        groups = [{"L": case["L"], "T": case["T"], "n_walkers": case["walkers"]}]
    ctx = muca.Context(groups, seed=seed & 0x7FFFFFFF)
    st["ctx"] = ctx
    if kind == "disordered":
        ctx.set_bonds(0, wl.random_bonds(case["L"], wl.DISORDERED["j1"], wl.DISORDERED["j2"],
                                         seed))
        ctx.run_graph(1, 20)
    elif kind == "production":
        L, T, V = case["L"], case["T"], case["L"] ** 3
        if V * case["walkers"] <= 30_000_000:
            # weights of a finished iteration: the transition's slope and the
            # noise of some tens of counts per bin; walkers over both phases
            rng = np.random.default_rng(seed)
            ctx.set_lnW(0, -FIELDS[T] / T * np.arange(V + 1) + 0.1 * rng.normal(size=V + 1))
            ctx.set_state(0, _spins(L, T, case["walkers"], seed))
            ctx.sweep_iter(10)
        else:
            # too many spins to be set quickly: weights and walkers as a few
            # short iterations from the random start leave them
            ctx.run_graph(4, 50)
        ctx.reserve_timeseries(case["sweeps"])
    else:
        # in the middle of a weight iteration: some short iterations are done
        ctx.run_graph(3, max(2, min(50, int(2e6 / max(s["V"] for s in ctx.specs)))))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "reweight":
        out = muca.reweight(st["ej"], st["ed"], st["m"], st["lnW"], 0, st["beta"], st["V"],
                            st["grid"], case["precision"])
        if case["precision"] == 32:
            out = out.astype(np.float32)  # what a 32-bit result holds
        return {n: out[:, k] for k, n in enumerate(("E_J", "E_Delta", "C", "chi", "U4"))}
    if kind == "transition":
        d, de, c, ce, sub = muca.find_peak(st["ej"], st["ed"], st["lnW"], 0, st["beta"], st["lo"],
                                           st["hi"], n_jack=case["blocks"])
        q, qe, b, be, at, qsub = muca.equal_height(st["ed"], st["lnW"], 0, st["beta"],
                                                   st["split"], st["eq_lo"], st["eq_hi"],
                                                   n_jack=case["blocks"])
        # a value and its error belong together
        return {"delta_star": np.array([d, de]), "c_star": np.array([c, ce]),
                "delta_sets": sub[:, 0], "c_sets": sub[:, 1],
                "delta_eqh": np.array([q, qe]), "barrier": np.array([b, be]),
                "eqh_sets": qsub[:, 0], "barrier_sets": qsub[:, 1],
                "bins": np.array(at, dtype=np.int64)}
    ctx = st["ctx"]
    if kind == "production":
        ctx.reserve_timeseries(case["sweeps"])
        ctx.sweep_iter(case["sweeps"], record=True)
        return {"series": ctx.get_timeseries(0)}
    ctx.run_graph(1, case["sweeps"])
    groups = range(len(ctx.specs))
    return {"lnW": [ctx.get_lnW(g) for g in groups],
            "flatness": np.array([ctx.get_flatness(g) for g in groups])}


# -------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind in ("reweight", "transition"):
        n, nE = case["walkers"] * case["samples"], case["L"] ** 3 + 1
        if kind == "reweight":
            # per bin and field: one exponential, counted as one operation, and
            # one multiply-add for each of the eight weighted sums
            return {"bytes": 12 * n + 8 * nE + 48 * case["grid"],
                    "flops": 17 * nE * case["grid"]}
        # per set, bisection step and bin: an exponential and five multiply-adds
        # (Delta*_L); a multiply-add and a comparison (equal height)
        return {"bytes": 8 * n + 4 * n + 16 * nE,
                "flops": (1 + case["blocks"]) * 63 * nE * (11 + 3)}
    if kind == "batch":
        sizes = [(s["L"] ** 3, s["n_walkers"]) for s in wl.mixed_groups(case["walkers"])]
    else:
        sizes = [(case["L"] ** 3, case["walkers"])]
    sites = sum(v * w for v, w in sizes)
    bins = sum(v + 1 for v, _ in sizes)
    # the lattices are read and written once (a pass keeps what fits on the
    # chip there), the weights and the histogram are read and written
    out = 12 * case["walkers"] * case["sweeps"] if kind == "production" else 16 * bins
    return {"bytes": 2 * sites + 8 * bins + out,
            "flops": OPS_PER_ATTEMPT * sites * case["sweeps"]}


# ------------------------------------------------------------------- exact
def _split_field(beta, delta):
    """beta delta as c1 + c2 with c1 E exact in 64 bits for every bin E."""
    c = Fraction(beta) * Fraction(float(delta))
    c1 = Fraction(round(c * (1 << 30)), 1 << 30)
    return float(c1), float(c - c1)


def _log_weights(c1, c2, E, lnW, star):
    """ln of the weights exp(-c E) / W(E) relative to bin star, per field (rows):
    the large terms are subtracted without rounding."""
    dE = E[None, :] - E[star][:, None]
    a, b = lnW[None, :], lnW[star][:, None]
    s = a - b
    t = s - a
    err = (a - (s - t)) - (b + t)
    main = -(c1[:, None] * dE) - s
    return main - (c2[:, None] * dE + err)


def _bins(e, n_e):
    return torch.bincount(e, minlength=n_e)


def _exact_reweight(st):
    beta, V = st["beta"], float(st["V"])
    lnW = torch.as_tensor(st["lnW"], device="cuda")
    nE = lnW.numel()
    E = torch.arange(nE, device="cuda", dtype=torch.float64)
    e = st["ed"].reshape(-1).long()
    n = _bins(e, nE).double()
    safe = n.clamp(min=1.0)

    def total(v):
        return torch.zeros(nE, device="cuda", dtype=torch.float64).index_add_(0, e, v)

    mej = total(st["ej"].reshape(-1).double()) / safe
    am = st["m"].reshape(-1).abs().double() / V
    cm = total(am) / safe
    vb = total((am - cm[e]) ** 2)
    q2, q4 = total(am ** 2), total(am ** 4)
    split = [_split_field(beta, d) for d in st["grid"]]
    c1 = torch.tensor([s[0] for s in split], device="cuda", dtype=torch.float64)
    c2 = torch.tensor([s[1] for s in split], device="cuda", dtype=torch.float64)
    out = []
    none = n == 0
    for k in range(0, len(split), 128):
        a, b = c1[k:k + 128], c2[k:k + 128]
        rough = -(a[:, None] * E[None, :]) - lnW[None, :]
        rough[:, none] = -float("inf")
        x = _log_weights(a, b, E, lnW, rough.argmax(1))
        x[:, none] = -float("inf")
        w = torch.exp(x)
        wn = w * n
        Z = wn.sum(1)
        mE, mJ, mu = (wn @ E) / Z, (wn @ mej) / Z, (wn @ cm) / Z
        m2, m4 = (w @ q2) / Z, (w @ q4) / Z
        cov = (wn * (mej[None, :] - mJ[:, None]) * (E[None, :] - mE[:, None])).sum(1) / Z
        var = (w * vb + wn * (cm[None, :] - mu[:, None]) ** 2).sum(1) / Z
        out.append(torch.stack([mJ, mE, -beta * cov, beta * V * var,
                                1.0 - m4 / (3.0 * m2 * m2)], 1))
    out = torch.cat(out).cpu().numpy()
    return {nm: out[:, k] for k, nm in enumerate(("E_J", "E_Delta", "C", "chi", "U4"))}


def _jackknife(x):
    w = len(x)
    return float(np.sqrt((w - 1) / w * np.sum((x - x.mean()) ** 2)))


def _exact_transition(st, blocks):
    beta = st["beta"]
    lnW = torch.as_tensor(st["lnW"], device="cuda")
    nE = lnW.numel()
    E = torch.arange(nE, device="cuda", dtype=torch.float64)
    rows = st["ed"].shape[0]
    cnt, sej = [], []
    for i in range(blocks):
        sl = slice(i * rows // blocks, (i + 1) * rows // blocks)
        e = st["ed"][sl].reshape(-1).long()
        cnt.append(_bins(e, nE))
        sej.append(torch.zeros(nE, device="cuda", dtype=torch.int64).index_add_(
            0, e, st["ej"][sl].reshape(-1).long()))
    cnt, sej = torch.stack(cnt), torch.stack(sej)
    n = torch.cat([cnt.sum(0)[None], cnt.sum(0)[None] - cnt]).double()
    mj = torch.cat([sej.sum(0)[None], sej.sum(0)[None] - sej]).double() / n.clamp(min=1.0)
    none = n == 0

    def moments(delta):
        sp = [_split_field(beta, d) for d in delta]
        c1 = torch.tensor([s[0] for s in sp], device="cuda", dtype=torch.float64)
        c2 = torch.tensor([s[1] for s in sp], device="cuda", dtype=torch.float64)
        rough = -(c1[:, None] * E[None, :]) - lnW[None, :]
        rough[none] = -float("inf")
        x = _log_weights(c1, c2, E, lnW, rough.argmax(1))
        x[none] = -float("inf")
        w = torch.exp(x) * n
        Z = w.sum(1)
        dj = mj - ((w * mj).sum(1) / Z)[:, None]
        dd = E[None, :] - ((w * E[None, :]).sum(1) / Z)[:, None]
        return (w * dj * dd).sum(1) / Z, (w * dj * dd * dd).sum(1) / Z

    lo, hi = np.full(len(n), st["lo"]), np.full(len(n), st["hi"])
    for _ in range(60):
        mid = lo + 0.5 * (hi - lo)
        up = moments(mid)[1].cpu().numpy() > 0
        lo, hi = np.where(up, mid, lo), np.where(up, hi, mid)
    d = lo + 0.5 * (hi - lo)
    c = -beta * moments(d)[0].cpu().numpy()

    lnn = torch.log(n)  # -inf where a bin is empty
    low = torch.arange(nE, device="cuda") < st["split"]

    def log_p(delta):
        bd = beta * torch.as_tensor(delta, device="cuda")
        return (lnn - bd[:, None] * E[None, :]) - lnW[None, :]

    def peaks(p):
        a = p.masked_fill(~low[None, :], -float("inf")).max(1)
        b = p.masked_fill(low[None, :], -float("inf")).max(1)
        return a, b

    lo, hi = np.full(len(n), st["eq_lo"]), np.full(len(n), st["eq_hi"])
    for _ in range(60):
        mid = lo + 0.5 * (hi - lo)
        a, b = peaks(log_p(mid))
        up = (a.values < b.values).cpu().numpy()
        lo, hi = np.where(up, mid, lo), np.where(up, hi, mid)
    q = lo + 0.5 * (hi - lo)
    p = log_p(q)
    a, b = peaks(p)
    i = torch.arange(nE, device="cuda")[None, :]
    between = (i >= a.indices[:, None]) & (i <= b.indices[:, None]) & ~none
    bottom = p.masked_fill(~between, float("inf")).min(1)
    top = torch.maximum(a.values, b.values)
    bar = ((top - bottom.values).cpu().numpy()) / (2.0 * beta * q)
    return {"delta_star": np.array([d[0], _jackknife(d[1:])]),
            "c_star": np.array([c[0], _jackknife(c[1:])]),
            "delta_sets": d[1:], "c_sets": c[1:],
            "delta_eqh": np.array([q[0], _jackknife(q[1:])]),
            "barrier": np.array([bar[0], _jackknife(bar[1:])]),
            "eqh_sets": q[1:], "barrier_sets": bar[1:], "bins": None}


def exact(case, seed):
    if case["kind"] == "reweight":
        return _exact_reweight(prepare(case, seed))
    if case["kind"] == "transition":
        return _exact_transition(prepare(case, seed), case["blocks"])
    return None
