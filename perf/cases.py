"""Performance cases of the Aggregate Risk Analysis engine.

Each case is work that a program using the engine has it do, through
``paper_1501_06326_gb300.ara.Ara``: pricing one layer and reading its PML and
TVaR, a layer with two-part secondary uncertainty, per-event output, a
portfolio of layers in one pass with and without the YET's event-major index,
a fresh YET indexed and priced, a pool of Event Loss Tables loaded and used, a
burst of served requests, and the tail figures of a Year Loss Table.

Inputs follow the seeded recipes of ``paper_1501_06326_gb300.synth`` (made
here on the GPU): trials of Poisson(lambda) events with uniform ids, records
with mean ~ LogNormal(10, 2), exposure = mean * U(2, 20) and sigma = mean *
U(0.1, 1) clipped so that both Beta shapes stay >= 0.05 (or the shapes
log-uniform in [0.2, 50], the stress recipe), and layer terms at percentiles
of the layer's own losses.  ``exact`` computes the same outputs in 64-bit
torch arithmetic of its own.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1501_06326_gb300 import ara

DEV = "cuda"
RPS = (100.0, 250.0)
EXACT_PAIRS = 200e6  # pairs that exact() inverts within about 20 seconds


# ------------------------------------------------------------------ the cases
def _layer(name, trials, events, catalogue, elts, entries, recipe="plain", correlated=0.0):
    return dict(name=name, kind="layer", trials=trials, events=events, catalogue=catalogue, elts=elts,
                entries=entries, recipe=recipe, correlated=correlated)


def listed():
    return [
        # the plain-1k configuration: the smallest call, a quick look at a small layer (launches and latency)
        _layer("layer-1k", 1_000, 100.0, 10_000, 3, 1_000),
        # an underwriter's first look at a contract: a ragged prefix of the full-size YET
        _layer("layer-20k", 20_011, 1000.0, 2_000_000, 15, 10_000),
        # the paper-shaped full analysis of one layer, the headline workload
        _layer("layer-1m", 1_000_000, 1000.0, 2_000_000, 15, 10_000),
        # a layer over 30 ELTs of one region's dense catalogue: most events held, several ELTs each
        _layer("layer-dense", 100_003, 250.0, 100_000, 30, 10_000),
        # records with a correlated part of sigma (Sections 3.1 and 3.2), stress-recipe Beta shapes
        _layer("xelt-300k", 300_000, 1000.0, 2_000_000, 15, 10_000, "stress", 0.5),
        # per-event rows for reports beyond the YLT (occurrence exceedance, event contributions)
        dict(name="events-200k", kind="events", trials=200_000, events=1000.0, catalogue=2_000_000, elts=15,
             entries=10_000, recipe="plain", correlated=0.0),
        # a portfolio of 16 uneven layers against a resident, indexed full-size YET
        dict(name="portfolio-1m", kind="portfolio", trials=1_000_000, events=1000.0, catalogue=2_000_000, pool=64,
             entries=10_000, layers=16, max_elts=32, index=True),
        # the same kind of portfolio priced once, on a YET without its index
        dict(name="portfolio-once", kind="portfolio", trials=150_001, events=1000.0, catalogue=2_000_000, pool=64,
             entries=10_000, layers=16, max_elts=32, index=False),
        # a new YET arrives: loaded, indexed and a portfolio priced on it
        dict(name="renewal-400k", kind="renewal", trials=400_000, events=1000.0, catalogue=2_000_000, pool=64,
             entries=10_000, layers=16, max_elts=32),
        # new ELTs arrive from a catastrophe model: loaded (Beta shapes, quantile tables) and a first layer priced
        dict(name="elts-150k", kind="pool", trials=10_000, events=1000.0, catalogue=2_000_000, elts=15,
             entries=10_000, recipe="plain", correlated=0.0),
        # a burst of pricing requests served against the resident YET and a pool of 200 ELTs
        dict(name="serve-128", kind="serve", trials=1_000_000, events=1000.0, catalogue=2_000_000, pool=200,
             entries=10_000, requests=128, max_elts=15),
        # the tail figures and the ranked trials of a full-size YLT
        dict(name="tail-1m", kind="tail", trials=1_000_003, rps=6, top=20_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "events", "portfolio", "portfolio", "renewal", "pool", "serve",
                       "tail"])
    if kind == "tail":
        return dict(kind=kind, trials=_log(rng, 1_000, 1_000_003), rps=rng.randint(1, 6), top=_log(rng, 10, 20_000))
    events = float(_log(rng, 50, 1_000))
    catalogue = _log(rng, 10_000, 2_000_000)
    if kind in ("layer", "events", "pool"):
        elts = rng.randint(1, 30)
        entries = _log(rng, 500, min(10_000, catalogue // 3))
        hits = elts * entries / catalogue  # ELT records held per event
        most = {"layer": 75e6, "events": 15e6, "pool": 5e6}[kind]  # lookups that find a record
        trials = _log(rng, 1_000, {"layer": 1_000_000, "events": 200_000, "pool": 20_000}[kind])
        trials = max(100, min(trials, int(most / (events * hits))))
        return dict(kind=kind, trials=trials, events=events, catalogue=catalogue, elts=elts, entries=entries,
                    recipe=rng.choice(["plain", "plain", "stress"]), correlated=rng.choice([0.0, 0.0, 0.5]))
    entries = _log(rng, 1_000, min(10_000, catalogue // 8))
    if kind == "serve":
        catalogue = max(catalogue, 400_000)
        return dict(kind=kind, trials=_log(rng, 50_000, 500_000), events=events, catalogue=catalogue,
                    pool=rng.randint(20, 200), entries=_log(rng, 1_000, catalogue // 200),
                    requests=_log(rng, 4, 128), max_elts=rng.randint(2, 15))
    pool, layers = rng.randint(8, 64), rng.randint(2, 32)
    most = 60e6 if kind == "renewal" or rng.random() < 0.5 else 150e6
    trials = max(1_000, min(_log(rng, 5_000, 400_000), int(most / (events * pool * entries / catalogue))))
    case = dict(kind=kind, trials=trials, events=events, catalogue=catalogue, pool=pool, entries=entries,
                layers=layers, max_elts=min(pool, 32))
    if kind == "portfolio":
        case["index"] = rng.random() < 0.5
    return case


# ------------------------------------------------------------------ inputs, made on the GPU from the seed
def _generator(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + stream) & 0x7FFFFFFFFFFF)
    return g


def _uniform(n, lo, hi, g):
    return lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)


def _yet(case, seed):
    """CSR Year Event Table: int64 offsets and int32 ids."""
    n, c = case["trials"], case["catalogue"]
    g = _generator(seed, 1)
    counts = torch.poisson(torch.full((n,), case["events"], device=DEV), generator=g).to(torch.int64)
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=off[1:])
    ids = torch.empty(int(off[-1]), dtype=torch.int32, device=DEV).random_(0, c, generator=g)
    return off, ids


def _pool(case, seed, n_elts):
    """A pool of ELTs in CSR form on the GPU (pool ids 0 .. n_elts - 1)."""
    g = _generator(seed, 2)
    n, c = case["entries"], case["catalogue"]
    ev = torch.cat([torch.randperm(c, generator=g, device=DEV)[:n].sort()[0] for _ in range(n_elts)]).to(torch.int32)
    r = n * n_elts
    mu = torch.exp(10.0 + 2.0 * torch.randn(r, generator=g, device=DEV, dtype=torch.float64))
    if case.get("recipe", "plain") == "stress":
        a = torch.exp(_uniform(r, math.log(0.2), math.log(50.0), g))
        b = torch.exp(_uniform(r, math.log(0.2), math.log(50.0), g))
        m = a / (a + b)
        ex = mu / m
        sg = ex * torch.sqrt(m * (1.0 - m) / (a + b + 1.0))
    else:
        ex = mu * _uniform(r, 2.0, 20.0, g)
        sg = mu * _uniform(r, 0.1, 1.0, g)
        m = mu / ex  # both Beta shapes stay at or above 0.05
        most = ex * torch.sqrt(m * (1.0 - m) / (1.0 + 0.05 / torch.minimum(m, 1.0 - m)))
        sg = torch.minimum(sg, most * (1.0 - 1e-6))
    sc = None
    if case.get("correlated", 0.0) > 0.0:
        sc = (sg * _uniform(r, 0.0, case["correlated"], g)).to(torch.float32)
        sg = sg - sc
    return dict(ids=np.arange(n_elts, dtype=np.int32), off=np.arange(n_elts + 1, dtype=np.int64) * n, ev=ev,
                mu=mu.to(torch.float32), sg=sg.to(torch.float32), ex=ex.to(torch.float32), sc=sc, n=n)


def _nearest_rank(sorted_values, pct):
    i = max(0, math.ceil(pct / 100.0 * sorted_values.numel()) - 1)
    return float(np.float32(sorted_values[i].item()))


def _terms(case, pool, elts, off, ids):
    """Layer terms at percentiles of the layer's primary-only losses: occurrence retention and limit at the
    50th and 99th of an event's loss, aggregate retention and limit at the 10th and 99th of a trial's."""
    table = torch.zeros(case["catalogue"], dtype=torch.float64, device=DEV)
    n = pool["n"]
    for j in elts:
        s = slice(j * n, (j + 1) * n)
        table[pool["ev"][s].long()] += pool["mu"][s].double()
    held = table[table > 0].sort()[0]
    occ_r, occ_l = _nearest_rank(held, 50.0), _nearest_rank(held, 99.0)
    t = min(case["trials"], 1_000)
    loss = (table[ids[: int(off[t])].long()] - occ_r).clamp(0.0, occ_l)
    trial = torch.repeat_interleave(torch.arange(t, device=DEV), off[1 : t + 1] - off[:t])
    sums = torch.zeros(t, dtype=torch.float64, device=DEV).index_add_(0, trial, loss).sort()[0]
    return occ_r, occ_l, _nearest_rank(sums, 10.0), max(_nearest_rank(sums, 99.0), 1.0)


def _inputs(case, seed):
    """The YET, the pool, the layers as (pool ids, terms) and, for served requests, their trial prefixes."""
    off, ids = _yet(case, seed)
    rng = np.random.default_rng([int(seed), 7])
    if case["kind"] in ("layer", "events", "pool"):
        pool = _pool(case, seed, case["elts"])
        sets = [list(range(case["elts"]))]
    else:
        pool = _pool(case, seed, case["pool"])
        count = case["requests"] if case["kind"] == "serve" else case["layers"]
        most = min(case["max_elts"], case["pool"])
        sets = [sorted(int(j) for j in rng.choice(case["pool"], int(rng.integers(1, most + 1)), replace=False))
                for _ in range(count)]
    layers = [(s, _terms(case, pool, s, off, ids)) for s in sets]
    lo, hi = math.log(min(10_000, case["trials"])), math.log(case["trials"])
    ends = [min(case["trials"], int(round(math.exp(rng.uniform(lo, hi))))) for _ in sets]
    return off, ids, pool, layers, ends


def _philox_seed(seed):
    return (int(seed) * 0x9E3779B97F4A7C15 + 0x1501) & 0xFFFFFFFFFFFFFFFF


def _ylt_input(case, seed):
    """A Year Loss Table as a layer gives it: some trials below the retention, some at the limit, the rest spread."""
    g = _generator(seed, 3)
    v = torch.exp(17.0 + 0.8 * torch.randn(case["trials"], generator=g, device=DEV, dtype=torch.float64))
    return (v - 1e7).clamp(0.0, 1.5e8)


def _row_capacity(case):
    """Rows a program makes room for: a tenth above the expected count (the rest stays as it was, zero)."""
    return int(1.1 * _expected_pairs(case)[1]) + 1_000


def _load_elts(eng, pool, host=None):
    p = host or pool
    if p["sc"] is not None:
        eng.load_xelts(p["ids"], p["off"], p["ev"], p["mu"], p["sg"], p["sc"], p["ex"])
    else:
        eng.load_elts(p["ids"], p["off"], p["ev"], p["mu"], p["sg"], p["ex"])


# ------------------------------------------------------------------ what a program has in hand before the call
def prepare(case, seed):
    kind = case["kind"]
    eng = ara.Ara(0)
    st = dict(kind=kind, eng=eng, seed=_philox_seed(seed), n=case["trials"])
    if kind == "tail":
        rps = np.array([10.0, 50.0, 100.0, 250.0, 500.0, 1000.0][: case["rps"]])
        n = case["trials"]
        st.update(ylt=_ylt_input(case, seed), rps=rps, top=min(case["top"], n),
                  values=torch.empty(min(case["top"], n), dtype=torch.float64, device=DEV),
                  trials=torch.empty(min(case["top"], n), dtype=torch.int64, device=DEV),
                  order=torch.empty(n, dtype=torch.int64, device=DEV))
        torch.cuda.synchronize()
        return st
    off, ids, pool, layers, ends = _inputs(case, seed)
    st.update(layers=layers, rps=np.array(RPS))
    torch.cuda.synchronize()
    if kind == "renewal":
        # a YET simulated on the device: it arrives there, its offsets on the host
        st.update(off=off.cpu().numpy(), ids=ids, catalogue=case["catalogue"])
    else:
        eng.load_yet(off.cpu().numpy(), ids, case["catalogue"])
    if kind == "pool":
        st["host"] = {k: (v.cpu().numpy() if isinstance(v, torch.Tensor) else v) for k, v in pool.items()}
    else:
        _load_elts(eng, pool)
    if kind == "serve" or case.get("index"):
        eng.build_yet_index()
    if kind == "serve":
        st["ends"] = ends
    else:
        st["ylt"] = torch.empty((len(layers), case["trials"]), dtype=torch.float64, device=DEV)
    if kind == "events":
        rows = _row_capacity(case)
        st["rows"] = dict(trial=torch.zeros(rows, dtype=torch.int64, device=DEV),
                          event_index=torch.zeros(rows, dtype=torch.int32, device=DEV),
                          event_id=torch.zeros(rows, dtype=torch.int32, device=DEV),
                          occ_loss=torch.zeros(rows, dtype=torch.float64, device=DEV),
                          agg_inc=torch.zeros(rows, dtype=torch.float64, device=DEV),
                          max_occ=torch.zeros(case["trials"], dtype=torch.float64, device=DEV))
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------ one pass, as a program calls the engine
def run(st):
    eng, kind, n = st["eng"], st["kind"], st["n"]
    if kind == "tail":
        pml, tvar = eng.pml_tvar(st["ylt"], st["rps"])
        values, trials = eng.top_m(st["ylt"], st["top"], 0, st["values"], st["trials"])
        order = eng.sort_ylt(st["ylt"], st["order"])
        return dict(pml=pml, tvar=tvar, values=values, trials=trials, order=order)
    if kind == "serve":
        tickets = [eng.submit(ids, terms, st["seed"], end, st["rps"])
                   for (ids, terms), end in zip(st["layers"], st["ends"])]
        done = [eng.wait(t, len(st["rps"])) for t in tickets]
        return dict(pml=np.stack([p for p, _ in done]), tvar=np.stack([t for _, t in done]))
    if kind == "portfolio":
        eng.run_layers(st["layers"], st["seed"], 0, n, st["ylt"])
        return dict(ylt=st["ylt"])
    if kind == "renewal":
        eng.load_yet(st["off"], st["ids"], st["catalogue"])
        eng.build_yet_index()
        eng.run_layers(st["layers"], st["seed"], 0, n, st["ylt"])
        return dict(ylt=st["ylt"])
    if kind == "pool":
        _load_elts(eng, None, st["host"])
    ids, terms = st["layers"][0]
    ylt = st["ylt"][0]
    if kind == "events":
        r = st["rows"]
        count = eng.run_layer_events(ids, terms, st["seed"], 0, n, ylt, r["trial"], r["event_index"], r["event_id"],
                                     r["occ_loss"], r["agg_inc"], r["max_occ"])
        pml, tvar = eng.pml_tvar(r["max_occ"], st["rps"])
        return dict(ylt=ylt, rows=r, count=count, pml=pml, tvar=tvar)
    eng.run_layer(ids, terms, st["seed"], 0, n, ylt)
    pml, tvar = eng.pml_tvar(ylt, st["rps"])
    return dict(ylt=ylt, pml=pml, tvar=tvar)


# ------------------------------------------------------------------ what a pass cannot do without
def _expected_pairs(case):
    """(events, distinct held events, lookups that find a record) expected of a pass."""
    e = case["trials"] * case["events"]
    n_elts = case.get("elts", case.get("pool"))
    p = case["entries"] / case["catalogue"]
    if case["kind"] in ("layer", "events", "pool"):
        return e, e * (1.0 - (1.0 - p) ** n_elts), e * n_elts * p
    if case["kind"] == "serve":
        lo, hi = min(10_000, case["trials"]), case["trials"]
        prefix = (hi - lo) / math.log(hi / lo) if hi > lo else hi  # mean of a log-uniform prefix
        pairs = case["requests"] * prefix * case["events"] * p * (1 + min(case["max_elts"], n_elts)) / 2
        return e, pairs, pairs
    used = n_elts * (1.0 - (1.0 - (1 + case["max_elts"]) / 2 / n_elts) ** case["layers"])
    return e, e * (1.0 - (1.0 - p) ** used), e * used * p


PAIR_FLOPS = 120.0  # the uniform (integer rounds), Phi^-1, a quantile and the terms


def work(case):
    kind, n = case["kind"], case["trials"]
    if kind == "tail":
        # the YLT read once for each of the three calls; ranked values, trials and the whole order written
        return {"bytes": 3 * 8.0 * n + 16.0 * min(case["top"], n) + 8.0 * n, "flops": 20.0 * n}
    e, held, pairs = _expected_pairs(case)
    records = 16.0 * case["entries"] * case.get("elts", case.get("pool"))
    yet = 4.0 * e + 8.0 * n
    flops = PAIR_FLOPS * pairs
    if kind == "serve":
        return {"bytes": records + 8.0 * held, "flops": flops}  # an occurrence is 8 bytes
    if kind == "portfolio":
        return {"bytes": records + 8.0 * n * case["layers"] + (8.0 * held if case["index"] else yet), "flops": flops}
    if kind == "renewal":  # the YET read, kept and indexed (8 bytes an occurrence)
        return {"bytes": records + 8.0 * n * case["layers"] + 2 * yet + 8.0 * e, "flops": flops}
    if kind == "pool":  # 16 bytes a record read, a quantile table of 32 nodes written and each node a root
        nodes = 32.0 * case["entries"] * case["elts"]
        return {"bytes": records + 16.0 * nodes + yet + 8.0 * n, "flops": flops + 1000.0 * nodes}
    if kind == "events":
        return {"bytes": records + yet + 16.0 * n + 32.0 * held, "flops": flops}
    return {"bytes": records + yet + 8.0 * n, "flops": flops}


# ------------------------------------------------------------------ the outputs in 64 bits
def _log_beta(a, b):
    return torch.lgamma(a) + torch.lgamma(b) - torch.lgamma(a + b)


def _fraction(a, b, x):
    """The continued fraction of I_x(a, b) (Abramowitz & Stegun 26.5.8), modified Lentz."""
    tiny = 1e-300
    guard = lambda v: torch.where(v.abs() < tiny, torch.full_like(v, tiny), v)
    qab, qap, qam = a + b, a + 1.0, a - 1.0
    c = torch.ones_like(a)
    d = 1.0 / guard(1.0 - qab * x / qap)
    h = d.clone()
    for m in range(1, 3_000):
        m2 = 2.0 * m
        t = m * (b - m) * x / ((qam + m2) * (a + m2))
        d = 1.0 / guard(1.0 + t * d)
        c = guard(1.0 + t / c)
        h = h * (d * c)
        t = -(a + m) * (qab + m) * x / ((a + m2) * (qap + m2))
        d = 1.0 / guard(1.0 + t * d)
        c = guard(1.0 + t / c)
        step = d * c
        h = h * step
        if m % 8 == 0 and float((step - 1.0).abs().max()) < 1e-14:
            break
    return h


def _log_cdf(a, b, lnb, r):
    """ln I_r(a, b) and its slope in ln r."""
    lower = r < (a + 1.0) / (a + b + 2.0)
    front = a * torch.log(r) + b * torch.log1p(-r) - lnb
    p, q, y = torch.where(lower, a, b), torch.where(lower, b, a), torch.where(lower, r, 1.0 - r)
    cf = _fraction(p, q, y) / p
    ln_i = torch.where(lower, front + torch.log(cf), torch.log1p(-torch.exp(front) * cf))
    return ln_i, torch.exp(front - ln_i) / (1.0 - r)


def _solve(a, b, ln_p):
    """r with ln I_r(a, b) = ln_p, r at most about 1/2: bracketed Newton (with Halley's term) in ln r."""
    lnb = _log_beta(a, b)
    out = torch.empty_like(a)
    live = torch.arange(a.numel(), device=a.device)
    lo = torch.full_like(a, -700.0)
    hi = torch.full_like(a, math.log(0.5) + 1e-9)
    u = ((ln_p + torch.log(a) + lnb) / a).clamp(-690.0, -1.0)
    for _ in range(80):
        r = torch.exp(u)
        ln_i, g = _log_cdf(a, b, lnb, r)
        f = ln_i - ln_p
        lo, hi = torch.where(f < 0, u, lo), torch.where(f < 0, hi, u)
        newton = -f / g
        curve = a - (b - 1.0) * r / (1.0 - r) - g
        den = 1.0 + 0.5 * newton * curve
        du = torch.where((den > 0.5) & (den < 2.0), newton / den, newton)
        un = u + du
        bad = ~((un > lo) & (un < hi))
        un = torch.where(bad & (du.abs() > 1e-9), 0.5 * (lo + hi), torch.where(bad, u, un))
        done = ((un - u).abs() < 1e-12) | (du.abs() < 1e-12)
        out[live] = un
        keep = ~done
        if not bool(keep.any()):
            break
        live, a, b, lnb, ln_p = live[keep], a[keep], b[keep], lnb[keep], ln_p[keep]
        lo, hi, u = lo[keep], hi[keep], un[keep]
    return torch.exp(out)


def _uniform_of(seed, trial, k, elt):
    """((w >> 9) + 1/2) 2^-23 with w word 0 of Philox4x32-10, counter (trial, k, elt, trial >> 32)."""
    m32 = 0xFFFFFFFF
    c0, c1, c2, c3 = trial & m32, k, elt, trial >> 32
    k0, k1 = seed & m32, seed >> 32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & m32) ^ c1 ^ k0), p1 & m32, (((p0 >> 32) & m32) ^ c3 ^ k1), p0 & m32
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return ((c0 >> 9).double() + 0.5) * 2.0**-23


class _Exact:
    """Losses of (event, ELT) pairs of a pool in 64 bits."""

    def __init__(self, case, pool, seed):
        self.seed, self.n = _philox_seed(seed), pool["n"]
        mu, ex, sg = pool["mu"].double(), pool["ex"].double(), pool["sg"].double()
        self.w = None
        if pool["sc"] is not None:
            sc = pool["sc"].double()
            nrm = torch.sqrt(sg * sg + sc * sc)
            self.w = sg / nrm, sc / nrm, sc > 0
            sg = sg + sc
        m = mu / ex
        most = torch.sqrt(m * (1.0 - m))
        s = torch.minimum(sg / ex, (1.0 - 1e-6) * most)
        nu = (most / s) ** 2 - 1.0
        self.a, self.b, self.ex = m * nu, (1.0 - m) * nu, ex
        ln_h, _ = _log_cdf(self.a, self.b, _log_beta(self.a, self.b), torch.full_like(m, 0.5))
        self.half = torch.exp(ln_h)
        self.where = pool["ev"].long()
        self.catalogue = case["catalogue"]

    def table(self, j):
        t = torch.full((self.catalogue,), -1, dtype=torch.int32, device=DEV)
        s = slice(j * self.n, (j + 1) * self.n)
        t[self.where[s]] = torch.arange(s.start, s.stop, dtype=torch.int32, device=DEV)
        return t

    def loss(self, rec, trial, k):
        """Losses of the pairs of pool records `rec`, those with like Beta shapes solved together."""
        out = torch.empty(rec.numel(), dtype=torch.float64, device=DEV)
        order = (self.a + self.b)[rec].argsort()
        for part in order.split(2_000_000):
            out[part] = self._loss(rec[part], trial[part], k[part])
        return out

    def _loss(self, r, trial, k):
        elt = torch.div(r, self.n, rounding_mode="floor")
        z = _uniform_of(self.seed, trial, k, elt)
        zc = 1.0 - z
        if self.w is not None:
            ze = _uniform_of(self.seed, trial, k, torch.full_like(elt, 0xFFFFFFFF))
            v = self.w[0][r] * torch.special.ndtri(z) + self.w[1][r] * torch.special.ndtri(ze)
            both = self.w[2][r]
            z, zc = (torch.where(both, torch.special.ndtr(v), z), torch.where(both, torch.special.ndtr(-v), zc))
        a, b = self.a[r], self.b[r]
        low = z <= self.half[r]
        root = _solve(torch.where(low, a, b), torch.where(low, b, a), torch.log(torch.where(low, z, zc)))
        return self.ex[r] * torch.where(low, root, 1.0 - root)


def _ranks(n, rps):
    return [min(n, max(1, math.ceil(n / rp))) for rp in rps]


def _tail(ylt, rps):
    top = ylt.sort(descending=True)[0]
    m = _ranks(ylt.numel(), rps)
    return (np.array([float(top[i - 1]) for i in m]), np.array([float(top[:i].mean()) for i in m]))


def _exact_layers(case, seed, inputs, want_rows=False):
    """Year losses of every layer, in 64 bits, trials in chunks; with want_rows the first layer's rows."""
    off, ids, pool, layers, _ = inputs
    ex = _Exact(case, pool, seed)
    n = case["trials"]
    ylt = torch.zeros((len(layers), n), dtype=torch.float64, device=DEV)
    used = sorted({j for s, _ in layers for j in s})
    tables = {j: ex.table(j) for j in used}
    rows = []
    density = case["entries"] / case["catalogue"]
    per_trial = case["events"] * max(1.0, len(layers) / 2, 12.0 * len(used) * density)
    step = max(1, int(40e6 / per_trial))
    for t0 in range(0, n, step):
        t1 = min(n, t0 + step)
        e0, e1 = int(off[t0]), int(off[t1])
        part = ids[e0:e1].long()
        trial = torch.repeat_interleave(torch.arange(t0, t1, device=DEV), off[t0 + 1 : t1 + 1] - off[t0:t1])
        k = torch.arange(e0, e1, device=DEV) - off[trial]
        g = torch.zeros((len(layers), e1 - e0), dtype=torch.float64, device=DEV)
        held = torch.zeros(e1 - e0, dtype=torch.bool, device=DEV) if want_rows else None
        at = [(tables[j][part] >= 0).nonzero()[:, 0] for j in used]
        rec = torch.cat([tables[j][part[x]] for j, x in zip(used, at)]).long()
        every = torch.cat(at)
        losses = ex.loss(rec, trial[every], k[every]).split([x.numel() for x in at])
        for j, x, loss in zip(used, at, losses):
            if want_rows:
                held[x] = True
            for i, (s, _) in enumerate(layers):
                if j in s:
                    g[i, x] += loss
        for i, (_, (occ_r, occ_l, agg_r, agg_l)) in enumerate(layers):
            o = (g[i] - occ_r).clamp(0.0, occ_l)
            total = torch.zeros(t1 - t0, dtype=torch.float64, device=DEV).index_add_(0, trial - t0, o)
            ylt[i, t0:t1] = (total - agg_r).clamp(0.0, agg_l)
            if want_rows:
                run_sum = torch.cumsum(o, 0)
                base = torch.cat([run_sum.new_zeros(1), run_sum])[off[trial] - e0]
                after = (run_sum - base - agg_r).clamp(0.0, agg_l)
                before = (run_sum - o - base - agg_r).clamp(0.0, agg_l)
                x = held.nonzero()[:, 0]
                most = torch.zeros(t1 - t0, dtype=torch.float64, device=DEV)
                most.scatter_reduce_(0, trial[x] - t0, o[x], "amax")
                rows.append((o[x], (after - before)[x], most))
    return ylt, rows


def exact(case, seed):
    kind = case["kind"]
    if kind == "tail":
        ylt = _ylt_input(case, seed)
        rps = [10.0, 50.0, 100.0, 250.0, 500.0, 1000.0][: case["rps"]]
        pml, tvar = _tail(ylt, rps)
        values = ylt.sort(descending=True)[0][: min(case["top"], case["trials"])]
        return dict(pml=pml, tvar=tvar, values=values, trials=None, order=None)
    if _expected_pairs(case)[2] > EXACT_PAIRS:
        return None
    inputs = _inputs(case, seed)
    if kind == "serve":  # one pass over all requests' layers; a request's year losses are its prefix
        ylt, _ = _exact_layers(case, seed, inputs)
        both = [_tail(ylt[i, :end], RPS) for i, end in enumerate(inputs[4])]
        return dict(pml=np.stack([p for p, _ in both]), tvar=np.stack([t for _, t in both]))
    ylt, rows = _exact_layers(case, seed, inputs, kind == "events")
    if kind in ("portfolio", "renewal"):
        return dict(ylt=ylt)
    if kind == "events":
        occ, inc, most = (torch.cat([r[i] for r in rows]) for i in range(3))
        room = torch.zeros((2, _row_capacity(case)), dtype=torch.float64, device=DEV)
        count = min(occ.numel(), room.shape[1])
        room[0, :count], room[1, :count] = occ[:count], inc[:count]
        pml, tvar = _tail(most, RPS)
        return dict(ylt=ylt[0], rows=dict(trial=None, event_index=None, event_id=None, occ_loss=room[0],
                                          agg_inc=room[1], max_occ=most), count=None, pml=pml, tvar=tvar)
    pml, tvar = _tail(ylt[0], RPS)
    return dict(ylt=ylt[0], pml=pml, tvar=tvar)
