"""Analyses and per-occurrence outputs over marked events against the same
calls over every row, in a context whose memory budget has no room for marks,
and against the oracle.

FP64 and Kahan trial losses agree bit for bit, and so does every
per-occurrence output (both forms sum exactly); FP32 losses in FP64 sums are
exact over marked events and round each addition over every row: within
events * 2^-52 of the total."""
import math

import numpy as np
import pytest

import workloads as W
from gpu_support import RTOL, mixed_check, running_bound, trial_bound

pytestmark = pytest.mark.gpu
INF = math.inf


@pytest.fixture(scope="module")
def are():
    import torch
    assert torch.cuda.is_available()
    import paper_1308_2066_gb300 as are
    are.lib()
    return are


# (ELTs, catalog, entries per ELT, retention, events a trial, ragged, FP32 rows,
# FP64 rows): every row format, trials of one pass of 512 events, of its
# quarters and of several passes, a catalog whose marks fold
CASES = [
    (6, 9000, 500, 2e5, 100, False, (32, False), (32, True)),
    (8, 9000, 900, 4e5, 513, True, (32, False), (64, True)),
    (12, 20_000, 700, 2e5, 1100, True, (32, True), (32, True)),
    (12, 900, 250, 1.1e6, 385, False, (64, False), (64, True)),
    (20, 900, 130, 1e6, 700, True, (64, True), (64, True)),
    (24, 3000, 120, 3e5, 1025, False, (32, True), (64, True)),
    (16, 1_600_000, 40_000, 2e5, 600, True, (32, True), (32, True)),
]
N = 300


def workload(case):
    """Trials few, some and most of whose events have a loss, whatever the
    catalog's share; the layer's aggregate terms take part."""
    J, C, nnz, occ_r, k, ragged, _, _ = case
    g = np.random.Generator(np.random.PCG64(5000 + J + k))
    shared = g.permutation(C)[:20]           # events of every ELT: rows past their inline terms
    elts = []
    for _ in range(J):
        ids = np.unique(np.concatenate([shared, g.permutation(C)[:nnz]])).astype(np.int32)
        elts.append(W.ELT(ids, g.lognormal(11, 1.5, ids.size)))
    loss = np.zeros(C)
    for e in elts:
        loss[e.ids] += e.losses
    some = np.flatnonzero(loss > occ_r)
    assert 0.005 < some.size / C < 0.4       # well below every limit for marks
    counts = g.poisson(k, N) if ragged else np.full(N, k)
    if ragged:
        counts[5] = 0
    ids = g.integers(0, C, counts.sum())
    most = np.repeat(g.choice([0.0, 0.3, 0.95], N), counts)
    ids = np.where(g.random(ids.size) < most, some[g.integers(0, some.size, ids.size)], ids).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    yet = W.YET(C, N, ids, None, off) if ragged else W.YET(C, N, ids, k)
    scale = float(np.mean(loss[some] - occ_r))
    return W.Workload("marked", yet, elts, [W.Layer(list(range(J)), occ_r, 20 * scale, 3 * scale, 200 * scale)])


def run(are, wl, precisions, rows, room):
    """{precision: (YLT, marginals, largest losses, YLT of those)}, the memory
    held."""
    import torch
    y, L = wl.yet, wl.layers[0]
    ctx = are.are_create(0, room)
    try:
        yet = are.are_load_yet(ctx, y.catalog, N, y.offsets, y.k or 0, y.ids)
        hs = [are.are_load_elt(ctx, e.ids, e.losses) for e in wl.elts]
        layer = are.are_define_layer(ctx, hs, L.occ_r, L.occ_l, L.agg_r, L.agg_l)
        got = {}
        for p in precisions:
            assert are.are_layer_rows(ctx, layer, yet, p) == rows
            out = torch.full((N,), -1.0, dtype=torch.float64, device="cuda")
            are.are_simulate(ctx, layer, yet, 0, N, p, out)
            ylt = out.cpu().numpy()
            # marginals from 8 bytes past a 16-byte boundary on, with room about them
            buf = torch.full((y.n_events + 3,), -7.0, dtype=torch.float64, device="cuda")
            top = torch.full((N,), -7.0, dtype=torch.float64, device="cuda")
            are.are_simulate_occurrences(ctx, layer, yet, 0, N, p, buf[1:], top, out)
            assert buf[0] == -7 and torch.all(buf[1 + y.n_events:] == -7)
            marg = buf[1:1 + y.n_events].cpu().numpy()
            got[p] = (ylt, marg, top.cpu().numpy(), out.cpu().numpy())
            # a range of trials writes the same
            b, m = 37, 111
            first, last = y.bounds(b)[0], y.bounds(b + m - 1)[1]
            buf.fill_(-7.0)
            are.are_simulate_occurrences(ctx, layer, yet, b, m, p, buf, top[:m], out[:m])
            assert torch.all(buf[last - first:] == -7)
            for part, whole in ((buf[:last - first], marg[first:last]), (top[:m], got[p][2][b:b + m]),
                                (out[:m], got[p][3][b:b + m])):
                np.testing.assert_array_equal(part.cpu().numpy(), whole)
        return got, are.are_memory_used(ctx)
    finally:
        are.are_destroy(ctx)


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"j{c[0]}_c{c[1]}_k{c[4]}")
def test_marked_events_against_every_row(are, orc, case):
    wl = workload(case)
    ref = orc.simulate_layer(wl, 0, marginals=True)
    bound = trial_bound(wl, 0)
    words = (wl.yet.catalog + 127) // 128 * 4
    marks = 4 * (words if words <= 41600 else 41600)
    for precisions, rows in (((0,), case[7]), ((1, 2), case[6])):
        got, held = run(are, wl, precisions, rows, 0)
        every, without = run(are, wl, precisions, rows, held - 4)
        assert without == held - marks           # no marks there: every row read
        for p in precisions:
            ylt, marg, top, trial = got[p]
            for a, b in zip(got[p][1:], every[p][1:]):
                np.testing.assert_array_equal(a, b)
            if p == 2:
                assert np.all(np.abs(ylt - every[p][0]) <= wl.yet.counts() * 2.0 ** -52 * bound)
            else:
                np.testing.assert_array_equal(ylt, every[p][0])
            for g, r, b in ((ylt, ref.ylt, bound), (trial, ref.ylt, bound), (top, ref.occ_max, bound),
                            (marg, ref.marginals, running_bound(wl, 0))):
                ok, st = mixed_check(g, r, b, RTOL[p])
                assert ok, (p, st)
