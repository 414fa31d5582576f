"""Kahan sums over marked events add a trial's losses as the every-row kernel
does in its default form, one group of 32 events per batch: the same bits, also
over 64-byte rows and trials of an odd number of groups."""
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


# (ELTs, entries per ELT, FP32 rows) over 900 events: dense and packed 64-byte
# rows, and 32-byte ones.  About a third of the events pass the retention, by
# losses over so wide a range that the last bits of a sum tell its order.
@pytest.mark.parametrize("k", [96, 160, 545])        # 3, 5 and 18 groups
@pytest.mark.parametrize("J,nnz,rows", [(12, 250, (64, False)), (20, 130, (64, True)), (12, 120, (32, True))])
def test_kahan_sums_of_marked_events_are_the_default_form(are, tmp_path, J, nnz, rows, k):
    import torch
    g = np.random.Generator(np.random.PCG64(700 + J + k))
    C, n = 900, 20_000
    yet = W.yet_fixed(g, n, k, C, timestamps=False)
    elts = [W.elt_lognormal(g, C, nnz, 5.0, 5.0) for _ in range(J)]
    for e in elts:
        e.losses[g.random(nnz) < 0.85] = 1e-6
    ctx = are.are_create(0)
    try:
        y = are.are_load_yet(ctx, C, n, None, k, yet.ids)
        hs = [are.are_load_elt(ctx, e.ids, e.losses) for e in elts]
        layer = are.are_define_layer(ctx, hs, 1e-4, INF, 0.0, INF)
        assert are.are_layer_rows(ctx, layer, y, 1) == rows

        def run():
            out = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
            are.are_simulate(ctx, layer, y, 0, n, 1, out)
            return out.cpu().numpy()

        got = run()
        path = tmp_path / "every_row.jsonl"
        path.write_text("".join(json.dumps({"key": f"p1_fixed_jp{jp}_ev{1 << b}_single", "kernel": 2, "rows_in_flight": 1,
                                            "trials_per_item": 8, "blocks_per_sm": 0, "ms": 1.0}) + "\n"
                                for jp in (8, 16, 32) for b in range(5, 12)))
        are.are_tune_load(ctx, str(path))
        assert (got > 0).mean() > 0.9
        np.testing.assert_array_equal(got, run())
    finally:
        are.are_destroy(ctx)
