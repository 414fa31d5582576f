"""The analysis over marked events (the default where a layer's events with
an occurrence loss are few) against the analysis that reads every row.

Both form an occurrence loss from the same row in the same arithmetic, and an
event without a mark adds 0.  FP32 with Kahan sums adds a trial's losses in
the same order, so the two agree bit for bit; FP64 sums are exact in both.
FP32 with FP64 sums is exact over marked events and rounds every addition (at
most `events` of them, and 5 in the merge) over all of them: within events *
2^-52 of the total."""
import json
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
INF = math.inf


@pytest.fixture(scope="module")
def are():
    import torch
    assert torch.cuda.is_available()
    import paper_1308_2066_gb300 as are
    are.lib()
    return are


# (ELTs, catalog, events a trial, ragged, entries per ELT, neutral terms):
# trials at and around a pass of 512 events and its quarters, rows of 32 and
# 64 bytes with overflows, more marks in a pass than its list holds, a catalog
# whose marks fold
CASES = [
    (4, 5000, 96, False, 300, True),
    (8, 40_000, 1000, False, 2000, False),
    (12, 40_000, 700, True, 1500, False),
    (16, 60_000, 511, False, 1500, True),
    (16, 60_000, 512, False, 1500, False),
    (16, 60_000, 513, False, 1500, True),
    (20, 30_000, 129, True, 700, True),
    (16, 3000, 1025, False, 130, True),
    (32, 20_000, 640, True, 300, True),
    (16, 1_600_000, 1100, True, 40_000, True),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"j{c[0]}_c{c[1]}_k{c[2]}")
def test_marked_events_equal_every_row(are, tmp_path, case):
    import torch
    J, C, k, ragged, nnz, neutral = case
    g = np.random.Generator(np.random.PCG64(4000 + J + k))
    n = 1501
    yet = W.yet_poisson(g, n, k, C, timestamps=False) if ragged else W.yet_fixed(g, n, k, C, timestamps=False)
    shared = g.permutation(C)[:20]           # events of every ELT: rows past their inline terms
    elts = []
    for _ in range(J):
        ids = np.unique(np.concatenate([shared, g.permutation(C)[:nnz]])).astype(np.int32)
        elts.append(W.ELT(ids, 100.0 * (1.0 - g.random(ids.size)) ** (-1.0 / 1.3)))
    terms = (0.0, INF, 0.0, INF) if neutral else (500.0, 5e5, 1e3, 1e7)
    ctx = are.are_create(0)
    try:
        y = are.are_load_yet(ctx, C, n, yet.offsets, yet.k or 0, yet.ids)
        hs = [are.are_load_elt(ctx, e.ids, e.losses) for e in elts]
        layer = are.are_define_layer(ctx, hs, *terms)

        def run(p, begin=0, m=n):
            out = torch.full((m,), -1.0, dtype=torch.float64, device="cuda")
            are.are_simulate(ctx, layer, y, begin, m, p, out)
            return out.cpu().numpy()

        for p in (0, 1, 2):
            got = run(p)
            assert (got > 0).mean() > 0.2
            parts = np.concatenate([run(p, b, m) for b, m in ((0, 1), (1, 700), (701, n - 701))])
            np.testing.assert_array_equal(parts, got)
            # every row read, with the default groups of 32 events for the row
            row_bytes, _ = are.are_layer_rows(ctx, layer, y, p)
            path = tmp_path / f"{p}.jsonl"
            keys = [f"p{p}_{'ragged' if ragged else 'fixed'}_jp{jp}_ev{1 << b}_single"
                    for jp in (4, 8, 12, 16, 20, 32) for b in range(5, 13)]
            path.write_text("".join(json.dumps(
                {"key": key, "kernel": 2, "rows_in_flight": 2 if p == 0 or row_bytes > 32 else 1,
                 "trials_per_item": 8, "blocks_per_sm": 0, "ms": 1.0}) + "\n" for key in keys))
            are.are_tune_load(ctx, str(path))
            want = run(p)
            if p == are.ARE_FP32_FP64AGG:
                most = np.diff(yet.offsets).max() if ragged else k
                np.testing.assert_allclose(got, want, rtol=float(most) * 2.0 ** -52, atol=0 if neutral else 1e-6)
            else:
                np.testing.assert_array_equal(got, want)
    finally:
        are.are_destroy(ctx)


def test_the_share_of_marked_events_decides(are):
    """An occurrence retention above every loss marks nothing, and a table
    built for one catalog serves another; both give the every-row results."""
    import torch
    g = np.random.Generator(np.random.PCG64(77))
    ctx = are.are_create(0)
    try:
        elts = [W.elt_lognormal(g, 4000, 3000) for _ in range(4)]
        hs = [are.are_load_elt(ctx, e.ids, e.losses) for e in elts]
        none = are.are_define_layer(ctx, hs, 1e300, INF, 0.0, INF)
        some = are.are_define_layer(ctx, hs, 2e6, INF, 0.0, INF)
        for C in (4000, 9000, 4000):
            yet = W.yet_fixed(g, 300, 200, C, timestamps=False)
            y = are.are_load_yet(ctx, C, 300, None, 200, yet.ids)
            out = torch.full((300,), -1.0, dtype=torch.float64, device="cuda")
            h = np.zeros(C)
            for e in elts:
                h[e.ids] += e.losses
            h = np.maximum(h - 2e6, 0.0)
            for p in (0, 1, 2):
                are.are_simulate(ctx, none, y, 0, 300, p, out)
                assert torch.all(out == 0)
                are.are_simulate(ctx, some, y, 0, 300, p, out)
                # a rounding of an event loss g scales by g, at most 1e8 here
                np.testing.assert_allclose(out.cpu().numpy(), h[yet.ids].reshape(300, 200).sum(1), rtol=1e-12 if p == 0 else 1e-5,
                                           atol=0 if p == 0 else 200 * 1e8 * 2.0 ** -23)
            are.are_free_yet(ctx, y)
    finally:
        are.are_destroy(ctx)


@pytest.mark.parametrize("J,C,nnz", [(3, 255, 100), (5, 256, 200), (9, 257, 100), (16, 513, 60), (16, 1000, 700),
                                     (32, 70_000, 700), (32, 300, 300), (10, 48 * 65536 * 4 + 300, 500)])
def test_rows_built_tile_by_tile(are, orc, J, C, nnz):
    """One-event trials give every event's loss from the rows as built: tiles
    of 256 events around their edges, more entries in a tile than it keeps
    between its passes, every ELT holding an event (overflows), ELTs whose
    last tile comes before the catalog's, an ELT without entries, and ids past
    the buckets.  FP64 and the folded table equal the oracle's bit for bit; FP32
    terms are rounded once and up to 32 of them added."""
    import torch
    g = np.random.Generator(np.random.PCG64(J + C))
    top = C if C < 1 << 20 else C - 1
    near = np.arange(top - 300, top) if C >= 1 << 20 else np.arange(C)
    elts = []
    for j in range(J):
        pool = near if j % 2 else near[: max(1, near.size - 40 * j % near.size)]
        ids = g.permutation(pool)[: min(nnz, pool.size)].astype(np.int32)
        elts.append(W.percentile_terms(W.ELT(ids, g.lognormal(11, 1.5, ids.size))))
    elts[J // 2] = W.ELT(np.zeros(0, np.int32), np.zeros(0))
    events = g.permutation(near)[:2000].astype(np.int32)
    yet = W.YET(catalog=C, n_trials=events.size, ids=events, k=1)
    wl = W.Workload("t", yet, elts, [W.Layer(list(range(J)), 2e4, 1e6, 0.0, INF)])
    ref = orc.simulate_layer(wl).ylt
    ctx = are.are_create(0)
    try:
        y = are.are_load_yet(ctx, C, events.size, None, 1, events)
        hs = [are.are_load_elt(ctx, e.ids, e.losses, e.fx, e.ded, e.lim, e.share) for e in elts]
        layer = are.are_define_layer(ctx, hs, 2e4, 1e6, 0.0, INF)
        for p in (0, 1, 2):
            out = torch.full((events.size,), -1.0, dtype=torch.float64, device="cuda")
            are.are_simulate(ctx, layer, y, 0, events.size, p, out)
            if p == 0:
                np.testing.assert_array_equal(out.cpu().numpy(), ref)
            else:    # 34 roundings at the scale of the event loss, at most 32 limits
                bound = 34 * 2.0 ** -24 * sum(e.lim for e in elts if np.isfinite(e.lim))
                np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=1e-5, atol=bound)
        are.are_simulate_folded(ctx, layer, y, 0, events.size, out)      # the folded table's tiles
        np.testing.assert_array_equal(out.cpu().numpy(), ref)
    finally:
        are.are_destroy(ctx)
