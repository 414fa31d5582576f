"""The work that users of the library have it do, as measurable cases.

Every case goes through the public calls of ``paper_1308_2066_gb300`` with
synthetic inputs of the shapes that this repository's workloads use: Year
Event Tables of fixed or Poisson trials with uniform event ids, lognormal or
Pareto Event Loss Tables with percentile terms, and layer terms from neutral
to the paper-scale ones.  Inputs are drawn on the GPU from the seed alone.

``listed`` gives the cases, ``draw`` one more of the same ranges, ``prepare``
what a program holds before the call, ``run`` one pass, ``work`` the bytes and
operations a pass cannot do without, and ``exact`` the same results from plain
torch in 64 bits.
"""
import math

import numpy as np
import torch

import paper_1308_2066_gb300 as are

INF = math.inf
PERIODS = (100.0, 250.0)
LEVELS = (0.99,)
CURVE = (2.0, 5.0, 10.0, 50.0, 100.0, 250.0)     # an exceedance curve's points
CURVE_LEVELS = (0.95, 0.99)

# Occurrence retention and limit, aggregate retention and limit, and the ELT
# entries that a trial of the named shape meets (10,000 trials of 100 events
# over 4 ELTs; the paper-scale layer): a layer's aggregate terms are written
# for the number of losses its trials hold.
TERMS = {
    "small": (5e4, 2e6, 1e5, 1e7, 80.0),
    "paper": (5e5, 2e7, 1e6, 1e8, 320.0),
    "regional": (5e4, 4e6, 1e6, 4e8, 300.0),
    "neutral": (0.0, INF, 0.0, INF, 1.0),
}


def listed():
    return [
        # The smallest analysis: a few thousand entries, 10,000 trials of 100
        # events, on the default stream with results on the host.  Launches
        # and waits are most of it.
        dict(name="quote_10k_fp64", kind="layer", trials=10_000, events=100, ragged=False, catalog=10_000, elts=4,
             nnz=2_000, losses="lognormal", terms="small", precision="fp64", wait=True),
        # An underwriter's quote: one contract over 50,000 trials, priced
        # while on the phone, results on the host.
        dict(name="quote_50k_fp32", kind="layer", trials=50_000, events=1000, ragged=False, catalog=1_000_000, elts=8,
             nnz=20_000, losses="lognormal", terms="paper", precision="fp32_kahan", wait=True),
        # The paper-scale layer, 1,000,000 trials of 1000 events and 16 ELTs:
        # table, analysis and risk measures, queued on a stream, in the FP32
        # mode and in FP64.
        dict(name="layer_1m_fp32", kind="layer", trials=1_000_000, events=1000, ragged=False, catalog=1_000_000,
             elts=16, nnz=20_000, losses="lognormal", terms="paper", precision="fp32_kahan", wait=False),
        dict(name="layer_1m_fp64", kind="layer", trials=1_000_000, events=1000, ragged=False, catalog=1_000_000,
             elts=16, nnz=20_000, losses="lognormal", terms="paper", precision="fp64", wait=False),
        # Ragged trials over a 2,000,000-event catalog, 32 heavy-tailed ELTs
        # and no terms, so that every loss reaches the trial sum.
        dict(name="ragged_2m_catalog", kind="layer", trials=400_001, events=1000, ragged=True, catalog=2_000_000,
             elts=32, nnz=20_000, losses="pareto", terms="neutral", precision="fp32_fp64agg", wait=False),
        # A regional model: a small catalog that the layer's ELTs cover
        # several times over, odd trial counts, short ragged trials.
        dict(name="dense_20k_catalog", kind="layer", trials=99_999, events=120, ragged=True, catalog=20_000, elts=27,
             nnz=1_777, losses="lognormal", terms="regional", precision="fp32_kahan", wait=False),
        # A book of layers of 1 to 32 ELTs over one ragged YET: every table
        # rebuilt, one graph of all layers, batched risk measures.
        dict(name="portfolio_24_layers", kind="portfolio", trials=100_000, events=1000, catalog=1_000_000, layers=24,
             pool=96, max_elts=32, nnz=27_500, precision="fp32_kahan"),
        # Year-event loss table: every occurrence's marginal, each trial's
        # largest occurrence and its loss.
        dict(name="occurrences_200k_fp64", kind="occurrences", trials=200_000, events=1000, ragged=False,
             catalog=1_000_000, elts=16, nnz=20_000, losses="lognormal", terms="paper", precision="fp64"),
        # The folded-table form of the paper-scale layer.
        dict(name="folded_1m", kind="folded", trials=1_000_000, events=1000, ragged=False, catalog=1_000_000, elts=16,
             nnz=20_000, losses="lognormal", terms="paper"),
        # A YET that stays in (pinned) host memory, its ids packed in the 20
        # bits that the catalog needs.
        dict(name="streamed_200k_packed", kind="streamed", trials=200_000, events=1000, catalog=1_000_000, elts=16,
             nnz=20_000, losses="lognormal", terms="paper", precision="fp32_kahan"),
        # An exceedance curve read from a finished YLT.
        dict(name="measures_1m", kind="measures", trials=1_000_000, zeros=0.25, ties=0.02),
        # The pricing server: a burst of requests of 1 to 16 ELTs and 10,000
        # to 200,000 trials over a resident YET.
        dict(name="serving_burst", kind="serving", trials=200_000, events=1000, catalog=1_000_000, pool=48,
             nnz=20_000, requests=24),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "layer", "portfolio", "occurrences", "folded", "streamed",
                       "measures", "serving"])
    if kind == "measures":
        return dict(kind=kind, trials=_log(rng, 2_000, 2_000_000), zeros=round(rng.uniform(0.0, 0.6), 3),
                    ties=round(rng.uniform(0.0, 0.05), 3))
    events = _log(rng, 40, 1500)
    most = {"layer": 1_000_000_000, "portfolio": 60_000_000, "occurrences": 200_000_000, "folded": 1_000_000_000,
            "streamed": 200_000_000, "serving": 200_000_000}[kind]
    trials = _log(rng, 2_000, max(2_001, min(1_000_000, most // events)))
    catalog = _log(rng, 10_000, 2_000_000)
    if kind == "portfolio":
        return dict(kind=kind, trials=trials, events=events, catalog=catalog, layers=rng.randint(2, 24), pool=64,
                    max_elts=32, nnz=max(200, int(catalog * rng.uniform(0.005, 0.05))),
                    precision=rng.choice(["fp32_kahan", "fp32_kahan", "fp32_fp64agg", "fp64"]))
    if kind == "serving":
        return dict(kind=kind, trials=max(10_000, trials), events=events, catalog=catalog, pool=32,
                    nnz=max(200, int(catalog * rng.uniform(0.005, 0.05))), requests=rng.randint(4, 32))
    case = dict(kind=kind, trials=trials, events=events, catalog=catalog, elts=rng.randint(1, 32),
                nnz=max(100, int(catalog * math.exp(rng.uniform(math.log(0.005), math.log(0.1))))),
                losses=rng.choice(["lognormal", "lognormal", "pareto"]),
                terms=rng.choice(["paper", "regional", "neutral"]))
    if kind != "streamed":
        case["ragged"] = rng.random() < 0.5
    if kind != "folded":
        case["precision"] = rng.choice(["fp32_kahan", "fp32_kahan", "fp32_fp64agg", "fp64"])
    if kind == "layer":
        case["wait"] = rng.random() < 0.5
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _yet(case, g):
    """(ids, offsets or None): uniform ids; ragged trials hold Poisson counts."""
    n, k = case["trials"], case["events"]
    offsets = None
    total = n * k
    if case.get("ragged", case["kind"] == "portfolio"):
        counts = torch.poisson(torch.full((n,), float(k), device="cuda"), generator=g).to(torch.int64)
        offsets = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(counts, 0, out=offsets[1:])
        total = int(offsets[-1])
    ids = torch.randint(0, case["catalog"], (total,), generator=g, device="cuda", dtype=torch.int32)
    return ids, offsets


def _elt(case, g, nnz, losses):
    """(ids, losses, deductible, limit): the terms at the 10th and 99th percentile of the losses."""
    ids = torch.randperm(case["catalog"], generator=g, device="cuda", dtype=torch.int64)[:nnz].to(torch.int32)
    if losses == "pareto":
        u = 1.0 - torch.rand(nnz, generator=g, device="cuda", dtype=torch.float64)
        x = torch.clamp(100.0 * u ** (-1.0 / 1.3), max=1e9)
        return ids, x, 0.0, INF
    x = torch.exp(11.0 + 1.5 * torch.randn(nnz, generator=g, device="cuda", dtype=torch.float64))
    s = torch.sort(x).values
    n = x.numel()
    return ids, x, float(s[max(1, -(-n // 10)) - 1]), float(s[max(1, -(-99 * n // 100)) - 1])


def _terms(case):
    occ_r, occ_l, agg_r, agg_l, met = TERMS[case["terms"]]
    scale = case["events"] * case["elts"] * case["nnz"] / case["catalog"] / met
    return (occ_r, occ_l, agg_r * scale, agg_l * scale)


def _layer_inputs(case, seed):
    g = _generator(seed)
    elts = [_elt(case, g, case["nnz"], case["losses"]) for _ in range(case["elts"])]
    return elts, _terms(case), _yet(case, g)


def _portfolio_inputs(case, seed):
    """A pool of ELTs of varying size and layers of 1 .. max_elts of them with
    terms at percentiles of their losses."""
    g = _generator(seed)
    r = np.random.Generator(np.random.PCG64(seed))
    sizes = [max(50, int(case["nnz"] * r.uniform(0.2, 1.8))) for _ in range(case["pool"])]
    pool = [_elt(case, g, min(n, case["catalog"]), "lognormal") for n in sizes]
    layers = []
    for _ in range(case["layers"]):
        members = [int(m) for m in r.choice(case["pool"], size=int(r.integers(1, case["max_elts"] + 1)),
                                            replace=False)]
        s = torch.sort(torch.cat([pool[m][1] for m in members])).values
        occ_r = float(s[int(r.uniform(0.0, 0.5) * (s.numel() - 1))])
        occ_l = float(s[int(r.uniform(0.9, 1.0) * (s.numel() - 1))])
        layers.append((members, (occ_r, occ_l, occ_r * float(r.uniform(1, 10)), occ_l * float(r.uniform(1, 10)))))
    return pool, layers, _yet(case, g)


def _requests(case, seed):
    r = np.random.Generator(np.random.PCG64([seed, 1]))
    out = []
    for _ in range(case["requests"]):
        members = [int(m) for m in r.choice(case["pool"], size=int(r.integers(1, 17)), replace=False)]
        occ_r = 6e4 * float(r.uniform(0.5, 5.0))
        occ_l = occ_r * float(r.uniform(5.0, 50.0))
        n = int(round(math.exp(r.uniform(math.log(10_000), math.log(case["trials"] + 1)))))
        out.append((members, (occ_r, occ_l, occ_r * float(r.uniform(1, 4)), occ_l * float(r.uniform(2, 10))),
                    min(n, case["trials"])))
    return out


def _ylt(case, seed):
    g = _generator(seed)
    n = case["trials"]
    y = torch.exp(14.0 + 2.0 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64))
    u = torch.rand(n, generator=g, device="cuda")
    y[u < case["zeros"]] = 0.0
    y[u > 1.0 - case["ties"]] = 1e8              # trials at the aggregate limit
    return y


# ---------------------------------------------------------------------------
# what a program keeps
# ---------------------------------------------------------------------------

_shared = {}


def _context():
    if "ctx" not in _shared:
        _shared["ctx"] = are.are_create(0)
        _shared["stream"] = torch.cuda.Stream()
    return _shared["ctx"], _shared["stream"]


class _State:
    """Handles of one case's inputs and its output buffers."""

    def __init__(self, case, ctx, stream):
        self.case, self.ctx, self.stream = case, ctx, stream
        self.yet, self.elts, self.layers, self.server = None, [], [], False
        self.own_context = False

    def load(self, elts, layers, yet):
        case = self.case
        self.elts = [are.are_load_elt(self.ctx, i, x, 1.0, d, lim, 1.0) for i, x, d, lim in elts]
        self.layers = [are.are_define_layer(self.ctx, [self.elts[m] for m in members], *terms)
                       for members, terms in layers]
        if yet is not None:
            ids, offsets = yet
            self.yet = are.are_load_yet(self.ctx, case["catalog"], case["trials"], offsets,
                                        0 if offsets is not None else case["events"], ids)

    def __del__(self):
        try:
            if self.server:
                are.are_server_stop(self.ctx)
            if self.own_context:
                are.are_destroy(self.ctx)
                return
            for h in self.layers:
                are.are_free_layer(self.ctx, h)
            for h in self.elts:
                are.are_free_elt(self.ctx, h)
            if self.yet is not None:
                are.are_free_yet(self.ctx, self.yet)
        except Exception:
            pass      # the interpreter is going down


def _doubles(n):
    return torch.zeros(n, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    ctx, stream = _context()
    if kind == "serving":
        ctx = are.are_create(0)
    s = _State(case, ctx, stream)
    s.own_context = kind == "serving"
    if kind == "measures":
        s.ylt = _ylt(case, seed)
        s.pml, s.tvar = _doubles(len(CURVE)), _doubles(len(CURVE_LEVELS))
        torch.cuda.current_stream().synchronize()
        return s
    if kind == "portfolio":
        pool, layers, yet = _portfolio_inputs(case, seed)
        s.load(pool, layers, yet)
        s.ylts = [_doubles(case["trials"]) for _ in layers]
    elif kind == "serving":
        g = _generator(seed)
        pool = [_elt(case, g, case["nnz"], "lognormal") for _ in range(case["pool"])]
        s.load(pool, [], _yet(case, g))
        s.requests = [([s.elts[m] for m in members], terms, n) for members, terms, n in _requests(case, seed)]
        are.are_server_start(ctx, s.yet)
        s.server = True
    else:
        elts, terms, yet = _layer_inputs(case, seed)
        s.load(elts, [(range(len(elts)), terms)], None if kind == "streamed" else yet)
        s.ylt = _doubles(case["trials"])
        if kind == "streamed":
            s.bits = max(1, (case["catalog"] - 1).bit_length())
            host = yet[0].cpu()
            s.packed = torch.empty(are.packed_words(host.numel(), s.bits), dtype=torch.int32, pin_memory=True)
            are.are_pack_ids(ctx, host.numpy(), s.bits, s.packed.data_ptr())
        if kind == "occurrences":
            s.marginals, s.largest = _doubles(yet[0].numel()), _doubles(case["trials"])
        s.pml, s.tvar = _doubles(len(PERIODS)), _doubles(len(LEVELS))
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    case, ctx = s.case, s.ctx
    kind, n = case["kind"], case["trials"]
    prec = are.PRECISIONS[case.get("precision", "fp32_kahan")]
    if kind == "layer":
        layer = s.layers[0]
        if case["wait"]:           # a program that waits for each answer
            are.are_prepare(ctx, layer, s.yet, prec)
            are.are_simulate(ctx, layer, s.yet, 0, n, prec, s.ylt)
            pml, tvar = are.are_risk_measures(ctx, s.ylt, n, PERIODS, LEVELS)
            return {"ylt": s.ylt, "pml": pml, "tvar": tvar}
        are.are_prepare(ctx, layer, s.yet, prec, stream=s.stream)
        are.are_simulate(ctx, layer, s.yet, 0, n, prec, s.ylt, stream=s.stream)
        are.are_risk_measures(ctx, s.ylt, n, PERIODS, LEVELS, stream=s.stream, out=(s.pml, s.tvar))
        return {"ylt": s.ylt, "pml": s.pml, "tvar": s.tvar}
    if kind == "portfolio":
        for layer in s.layers:
            are.are_prepare(ctx, layer, s.yet, prec, stream=s.stream)
        are.are_simulate_portfolio(ctx, s.layers, s.yet, 0, n, prec, s.ylts, stream=s.stream)
        pml, tvar = are.are_risk_measures_batch(ctx, s.ylts, n, PERIODS, LEVELS, stream=s.stream)
        return {"ylts": list(s.ylts), "pml": pml, "tvar": tvar}
    if kind == "occurrences":
        are.are_prepare(ctx, s.layers[0], s.yet, prec, stream=s.stream)
        are.are_simulate_occurrences(ctx, s.layers[0], s.yet, 0, n, prec, s.marginals, s.largest, s.ylt,
                                     stream=s.stream)
        return {"marginals": s.marginals, "largest": s.largest, "ylt": s.ylt}
    if kind == "folded":
        are.are_prepare_folded(ctx, s.layers[0], s.yet, stream=s.stream)
        are.are_simulate_folded(ctx, s.layers[0], s.yet, 0, n, s.ylt, stream=s.stream)
        are.are_risk_measures(ctx, s.ylt, n, PERIODS, LEVELS, stream=s.stream, out=(s.pml, s.tvar))
        return {"ylt": s.ylt, "pml": s.pml, "tvar": s.tvar}
    if kind == "streamed":
        are.are_simulate_streamed_packed(ctx, s.layers[0], case["catalog"], n, None, case["events"],
                                         s.packed.data_ptr(), s.bits, prec, s.ylt, stream=s.stream)
        are.are_risk_measures(ctx, s.ylt, n, PERIODS, LEVELS, stream=s.stream, out=(s.pml, s.tvar))
        return {"ylt": s.ylt, "pml": s.pml, "tvar": s.tvar}
    if kind == "measures":
        are.are_risk_measures(ctx, s.ylt, n, CURVE, CURVE_LEVELS, stream=s.stream, out=(s.pml, s.tvar))
        return {"pml": s.pml, "tvar": s.tvar}
    tickets = [are.are_submit(ctx, members, *terms, trials, PERIODS, LEVELS) for members, terms, trials in s.requests]
    got = [are.are_wait(ctx, t) for t in tickets]
    return {"status": np.array([r["status"] for r in got], dtype=np.int64),
            "pml": np.array([r["pml"] for r in got]), "tvar": np.array([r["tvar"] for r in got])}


def work(case):
    """Each id and ELT entry (id and loss) read once, each result written once;
    an addition and a clamp per occurrence, the financial terms per entry."""
    n, kind = case["trials"], case["kind"]
    if kind == "measures":
        return {"bytes": 8.0 * n, "flops": 1.0 * n}
    occ = float(n) * case["events"]
    if kind == "serving":
        part = [(len(m), t) for m, _, t in _requests(case, 7)]
        occ = sum(t for _, t in part) * float(case["events"])
        entries = sum(j for j, _ in part) * float(case["nnz"])
        return {"bytes": 4.0 * occ + 12.0 * entries, "flops": 4.0 * occ + 5.0 * entries}
    if kind == "portfolio":
        entries = case["layers"] * 0.5 * (1 + case["max_elts"]) * case["nnz"]
        return {"bytes": 4.0 * occ + 12.0 * entries + 8.0 * n * case["layers"],
                "flops": 4.0 * occ * case["layers"] + 5.0 * entries}
    entries = float(case["elts"]) * case["nnz"]
    bits = max(1, (case["catalog"] - 1).bit_length()) if kind == "streamed" else 32
    out = 8.0 * n + (8.0 * n + 8.0 * occ if kind == "occurrences" else 0.0)
    return {"bytes": occ * bits / 8.0 + 12.0 * entries + out, "flops": 4.0 * occ + 5.0 * entries}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _event_losses(catalog, elts, terms):
    """Occurrence loss of every catalog event (0 past the catalog)."""
    h = torch.zeros(catalog + 1, dtype=torch.float64, device="cuda")
    for ids, x, ded, lim in elts:
        h[ids.long()] += torch.clamp(x - ded, min=0.0).clamp(max=lim)
    h = torch.clamp(h - terms[0], min=0.0).clamp(max=terms[1])
    h[catalog] = 0.0
    return h


def _blocks(case, yet, trials):
    """(first trial, id matrix) for blocks of trials, ragged ones padded with the id `catalog`."""
    ids, offsets = yet
    step = max(1, 40_000_000 // (2 * case["events"]))
    for t0 in range(0, trials, step):
        t1 = min(trials, t0 + step)
        if offsets is None:
            yield t0, ids[t0 * case["events"]: t1 * case["events"]].view(t1 - t0, case["events"]), None
            continue
        off = offsets[t0: t1 + 1]
        width = int((off[1:] - off[:-1]).max()) if t1 > t0 else 0
        at = off[:-1, None] + torch.arange(width, device="cuda")[None, :]
        inside = at < off[1:, None]
        block = torch.where(inside, ids[at.clamp(max=max(0, ids.numel() - 1))], case["catalog"])
        yield t0, block, inside


def _trial_losses(case, h, terms, yet, trials):
    out = _doubles(trials)
    for t0, block, _ in _blocks(case, yet, trials):
        total = h[block.long()].sum(1)
        out[t0: t0 + block.shape[0]] = torch.clamp(total - terms[2], min=0.0).clamp(max=terms[3])
    return out


def _measures(ylt, periods, levels):
    n = ylt.numel()
    s = torch.sort(ylt, descending=True).values
    pml = [float(s[(n * 1_000_000 + round(p * 1e6) - 1) // round(p * 1e6) - 1]) for p in periods]
    tvar = [float(s[: (n * (1_000_000_000 - round(a * 1e9)) + 999_999_999) // 1_000_000_000].mean()) for a in levels]
    return torch.tensor(pml, dtype=torch.float64), torch.tensor(tvar, dtype=torch.float64)


def exact(case, seed):
    kind, n = case["kind"], case["trials"]
    if kind == "measures":
        pml, tvar = _measures(_ylt(case, seed), CURVE, CURVE_LEVELS)
        return {"pml": pml, "tvar": tvar}
    if kind == "portfolio":
        pool, layers, yet = _portfolio_inputs(case, seed)
        ylts, pml, tvar = [], [], []
        for members, terms in layers:
            h = _event_losses(case["catalog"], [pool[m] for m in members], terms)
            ylts.append(_trial_losses(case, h, terms, yet, n))
            p, t = _measures(ylts[-1], PERIODS, LEVELS)
            pml.append(p)
            tvar.append(t)
        return {"ylts": ylts, "pml": torch.stack(pml), "tvar": torch.stack(tvar)}
    if kind == "serving":
        g = _generator(seed)
        pool = [_elt(case, g, case["nnz"], "lognormal") for _ in range(case["pool"])]
        yet = _yet(case, g)
        pml, tvar = [], []
        for members, terms, trials in _requests(case, seed):
            h = _event_losses(case["catalog"], [pool[m] for m in members], terms)
            p, t = _measures(_trial_losses(case, h, terms, yet, trials), PERIODS, LEVELS)
            pml.append(p)
            tvar.append(t)
        return {"status": None, "pml": torch.stack(pml), "tvar": torch.stack(tvar)}
    elts, terms, yet = _layer_inputs(case, seed)
    h = _event_losses(case["catalog"], elts, terms)
    if kind != "occurrences":
        ylt = _trial_losses(case, h, terms, yet, n)
        pml, tvar = _measures(ylt, PERIODS, LEVELS)
        return {"ylt": ylt, "pml": pml, "tvar": tvar}
    marginals, largest, ylt = [], _doubles(n), _doubles(n)
    for t0, block, inside in _blocks(case, yet, n):
        o = h[block.long()]
        a = torch.clamp(torch.cumsum(o, 1) - terms[2], min=0.0).clamp(max=terms[3])
        m = torch.diff(a, dim=1, prepend=torch.zeros_like(a[:, :1]))
        marginals.append(m.reshape(-1) if inside is None else m[inside])
        largest[t0: t0 + block.shape[0]] = o.amax(1)
        ylt[t0: t0 + block.shape[0]] = a[:, -1]
    return {"marginals": torch.cat(marginals), "largest": largest, "ylt": ylt}
