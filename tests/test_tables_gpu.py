"""A layer's tables over a context's life: what a call builds, leaves alone,
and does without where memory is short."""
import json
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
INF = math.inf
CATALOG = 30_000


@pytest.fixture(scope="module")
def are():
    import torch
    assert torch.cuda.is_available()
    import paper_1308_2066_gb300 as are
    are.lib()
    return are


def elts_of(J, nnz=400, seed=0):
    g = np.random.Generator(np.random.PCG64(900 + J + seed))
    return [W.ELT(g.permutation(CATALOG)[:nnz].astype(np.int32), g.lognormal(11, 1.5, nnz)) for _ in range(J)]


def load_elts(are, ctx, elts):
    return [are.are_load_elt(ctx, e.ids, e.losses) for e in elts]


def yet_of(are, ctx, n, k, seed):
    ids = np.random.Generator(np.random.PCG64(seed)).integers(0, CATALOG, n * k).astype(np.int32)
    return are.are_load_yet(ctx, CATALOG, n, None, k, ids)


def simulate(are, ctx, layer, y, n, p):
    import torch
    out = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
    are.are_simulate(ctx, layer, y, 0, n, p, out)
    return out.cpu().numpy()


# dense 32-byte rows and packed rows; FP32 with either sum reads the same rows
@pytest.mark.parametrize("J", [6, 12])
def test_a_table_that_is_there_is_only_read(are, J):
    """Once a layer's table is built, no analysis writes it again, whatever
    precision, trial length or call comes next: each is one kernel."""
    import torch
    n, k = 300, 200
    ctx, fresh = are.are_create(0), are.are_create(0)
    try:
        elts = elts_of(J)
        layer = are.are_define_layer(ctx, load_elts(are, ctx, elts), 3e4, 2e6, 0.0, INF)
        short, long_ = yet_of(are, ctx, n, 20, 1), yet_of(are, ctx, n, k, 2)
        other = are.are_define_layer(fresh, load_elts(are, fresh, elts), 3e4, 2e6, 0.0, INF)
        other_long = yet_of(are, fresh, n, k, 2)
        marg = torch.zeros(n * k, dtype=torch.float64, device="cuda")
        for first, later in ((1, (1, 2)), (0, (0,))):
            are.are_prepare(ctx, layer, short, first)
            simulate(are, ctx, layer, short, n, first)
            for p in later:
                for call in (lambda: simulate(are, ctx, layer, short, n, p),
                             lambda: simulate(are, ctx, layer, long_, n, p),
                             lambda: are.are_simulate_occurrences(ctx, layer, long_, 0, n, p, marg)):
                    before = are.are_launch_count(ctx)
                    call()
                    assert are.are_launch_count(ctx) == before + 1
                np.testing.assert_array_equal(simulate(are, ctx, layer, long_, n, p),
                                              simulate(are, fresh, other, other_long, n, p))
    finally:
        are.are_destroy(ctx)
        are.are_destroy(fresh)


@pytest.mark.parametrize("J,p", [(6, 1), (12, 2), (12, 0)])
def test_rows_without_room_for_their_marks(are, J, p):
    """A memory budget that holds a layer's rows but not their marks: the
    analysis reads every row instead, and the losses are the same."""
    n, k = 200, 150
    elts = elts_of(J)

    def run(room):
        ctx = are.are_create(0, room)
        try:
            y = yet_of(are, ctx, n, k, 3)
            layer = are.are_define_layer(ctx, load_elts(are, ctx, elts), 3e4, 2e6, 0.0, INF)
            loaded = are.are_memory_used(ctx)
            got = simulate(are, ctx, layer, y, n, p)
            np.testing.assert_array_equal(simulate(are, ctx, layer, y, n, p), got)
            return got, loaded, are.are_memory_used(ctx)
        finally:
            are.are_destroy(ctx)

    want, loaded, used = run(0)
    assert (want > 0).mean() > 0.2
    marks = (CATALOG + 127) // 128 * 16
    assert used - loaded >= CATALOG * 32 + marks
    got, _, held = run(used - marks // 2)
    assert held == used - marks
    if p == 2:      # the sums over every row round each addition
        np.testing.assert_allclose(got, want, rtol=k * 2.0 ** -52, atol=0)
    else:
        np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("p,kernel", [(1, 0), (1, 1), (2, 0), (2, 2), (0, 1), (0, 3)])
def test_a_portfolio_of_one_layer_under_a_tuned_choice(are, tmp_path, p, kernel):
    """A tuning entry for several layers also decides for a portfolio of one:
    its tables are the ones that the kernel reads, and the losses are those of
    are_simulate under the same choice."""
    import torch
    n, k, J = 200, 150, 12
    elts = elts_of(J)
    got = {}
    for kind in ("multi", "single"):
        ctx = are.are_create(0)
        try:
            y = yet_of(are, ctx, n, k, 4)
            layer = are.are_define_layer(ctx, load_elts(are, ctx, elts), 3e4, 2e6, 0.0, INF)
            path = tmp_path / "tune.jsonl"
            path.write_text("".join(json.dumps(
                {"key": f"p{p}_fixed_jp{jp}_ev256_{kind}", "kernel": kernel, "rows_in_flight": 1,
                 "trials_per_item": 8, "blocks_per_sm": 0, "ms": 1.0}) + "\n" for jp in (12, 16)))
            are.are_tune_load(ctx, str(path))
            if kind == "single":
                got[kind] = simulate(are, ctx, layer, y, n, p)
            else:
                out = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
                are.are_simulate_portfolio(ctx, [layer], y, 0, n, p, [out])
                got[kind] = out.cpu().numpy()
        finally:
            are.are_destroy(ctx)
    assert (got["multi"] > 0).mean() > 0.2
    np.testing.assert_array_equal(got["multi"], got["single"])


@pytest.mark.parametrize("p", [1, 2])
def test_a_compact_layer_under_the_tuned_persistent_kernel(are, tmp_path, p):
    """The persistent kernel reads the dense table, which is then built for a
    layer of the compact layout too, and again for another catalog."""
    n, k, J = 200, 150, 12
    ctx = are.are_create(0)
    try:
        layer = are.are_define_layer(ctx, load_elts(are, ctx, elts_of(J)), 3e4, 2e6, 0.0, INF)
        path = tmp_path / "tune.jsonl"
        path.write_text(json.dumps({"key": f"p{p}_fixed_jp16_ev256_single", "kernel": 0, "rows_in_flight": 1,
                                    "trials_per_item": 8, "blocks_per_sm": 0, "ms": 1.0}) + "\n")
        are.are_tune_load(ctx, str(path))
        for catalog in (CATALOG, CATALOG + 5000):
            ids = np.random.Generator(np.random.PCG64(5)).integers(0, catalog, n * k).astype(np.int32)
            y = are.are_load_yet(ctx, catalog, n, None, k, ids)
            out = {}
            for layout in (are.ARE_LAYOUT_COMPACT, are.ARE_LAYOUT_DIRECT):
                are.are_set_table_layout(ctx, layer, layout)
                out[layout] = simulate(are, ctx, layer, y, n, p)
            assert (out[are.ARE_LAYOUT_DIRECT] > 0).mean() > 0.2
            np.testing.assert_array_equal(out[are.ARE_LAYOUT_COMPACT], out[are.ARE_LAYOUT_DIRECT])
    finally:
        are.are_destroy(ctx)


def test_the_batched_selection_within_a_budget(are):
    """Its scratch is charged to the budget, given back to whoever needs the
    room, and done without where there is none: the measures are the same."""
    import torch
    g = np.random.Generator(np.random.PCG64(8))
    ylts = [torch.from_numpy(g.lognormal(14, 2.0, 20_000)).cuda() for _ in range(5)]
    args = (ylts, 20_000, (100.0, 20.0), (0.99,))
    ctx = are.are_create(0)
    try:
        want = are.are_risk_measures_batch(ctx, *args)
        held = are.are_memory_used(ctx)
        assert held > 100_000
    finally:
        are.are_destroy(ctx)
    for room in (held, held // 2, 256):
        ctx = are.are_create(0, room)
        try:
            for _ in range(2):
                for a, b in zip(are.are_risk_measures_batch(ctx, *args), want):
                    np.testing.assert_array_equal(a, b)
                assert are.are_memory_used(ctx) <= room
            if room > 256:     # what the scratch holds is to be had
                are.are_load_yet(ctx, 10, 1, None, (room - 256) // 4 - 64, np.zeros((room - 256) // 4 - 64, np.int32))
                for a, b in zip(are.are_risk_measures_batch(ctx, *args), want):
                    np.testing.assert_array_equal(a, b)
        finally:
            are.are_destroy(ctx)


def test_a_refused_table_is_not_kept(are):
    """A layer whose ELT holds an id outside the YET's catalog is refused each
    time, in every form, and keeps no table."""
    import torch
    ctx = are.are_create(0)
    try:
        ids = np.array([3, 700], np.int32)
        layer = are.are_define_layer(ctx, [are.are_load_elt(ctx, ids, np.array([5.0, 7.0]))])
        y = are.are_load_yet(ctx, 700, 4, None, 8, np.full(32, 3, np.int32))
        out = torch.zeros(4, dtype=torch.float64, device="cuda")
        held = are.are_memory_used(ctx)
        for call in (lambda: are.are_prepare_folded(ctx, layer, y),
                     lambda: are.are_simulate_folded(ctx, layer, y, 0, 4, out),
                     lambda: are.are_prepare(ctx, layer, y, 0), lambda: are.are_prepare(ctx, layer, y, 1),
                     lambda: are.are_simulate(ctx, layer, y, 0, 4, 0, out),
                     lambda: are.are_simulate(ctx, layer, y, 0, 4, 1, out)):
            with pytest.raises(are.AreError) as e:
                call()
            assert e.value.status == are.ARE_EINVAL
            assert are.are_memory_used(ctx) == held
    finally:
        are.are_destroy(ctx)
