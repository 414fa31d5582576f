"""The register-rows kernels read one or two groups of 32 events at a time, by
default as the row's size calls for.  A lane gets the same events of a trial in
the same order either way, so the trial losses are the same bits; they match
the oracle."""
import json
import math

import numpy as np
import pytest

import workloads as W
from gpu_support import RTOL, mixed_check, trial_bound

pytestmark = pytest.mark.gpu
INF = math.inf


@pytest.fixture(scope="module")
def are():
    import torch
    assert torch.cuda.is_available()
    import paper_1308_2066_gb300 as are
    are.lib()
    return are


# (ELTs, entries per ELT, FP32 rows, FP64 rows) over 900 events: most events
# have a loss, so every row is read
ROWS = [(12, 250, (64, False), (64, True)), (20, 130, (64, True), (64, True)), (32, 120, (64, True), (64, True))]


@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("J,nnz,rows32,rows64", ROWS)
def test_groups_of_32_events(are, orc, tmp_path, J, nnz, rows32, rows64, ragged):
    import torch
    g = np.random.Generator(np.random.PCG64(400 + J + ragged))
    C, n = 900, 600
    if ragged:                      # empty trials, and lengths around one and two groups
        k = g.choice([0, 1, 31, 32, 33, 63, 64, 65, 96, 97, 200], n)
        off = np.concatenate([[0], np.cumsum(k)]).astype(np.int64)
        yet = W.YET(C, n, g.integers(0, C, off[-1]).astype(np.int32), None, off)
    else:
        yet = W.yet_fixed(g, n, 97, C, timestamps=False)
    elts = [W.elt_lognormal(g, C, nnz) for _ in range(J)]
    wl = W.Workload("groups", yet, elts, [W.Layer(list(range(J)), 0.0, INF, 0.0, INF)])
    ref = orc.simulate_layer(wl)
    ctx = are.are_create(0)
    try:
        y = are.are_load_yet(ctx, C, n, yet.offsets, yet.k or 0, yet.ids)
        hs = [are.are_load_elt(ctx, e.ids, e.losses, e.fx, e.ded, e.lim, e.share) for e in elts]
        layer = are.are_define_layer(ctx, hs, 0.0, INF, 0.0, INF)
        assert are.are_layer_rows(ctx, layer, y, 1) == rows32
        assert are.are_layer_rows(ctx, layer, y, 0) == rows64
        for p in (0, 1, 2):
            out = {}
            for groups in (0, 1, 2):
                path = tmp_path / f"{p}_{groups}.jsonl"
                path.write_text("".join(json.dumps(
                    {"key": f"p{p}_{'ragged' if ragged else 'fixed'}_jp{jp}_ev{1 << b}_single", "kernel": 2,
                     "rows_in_flight": groups, "trials_per_item": 8, "blocks_per_sm": 0, "ms": 1.0}) + "\n"
                    for jp in (12, 16, 20, 32) for b in range(5, 9)))
                are.are_tune_load(ctx, str(path))
                ylt = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
                are.are_simulate(ctx, layer, y, 0, n, p, ylt)
                out[groups] = ylt.cpu().numpy()
            np.testing.assert_array_equal(out[0], out[1])
            np.testing.assert_array_equal(out[0], out[2])
            ok, st = mixed_check(out[0], ref.ylt, trial_bound(wl, 0), RTOL[p])
            assert ok, (p, st)
    finally:
        are.are_destroy(ctx)
