"""Loading an ELT: the device memory it takes, what it waits for, and ELTs
whose entries found no room for their buckets' offsets."""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
INF = math.inf
CATALOG, N, K = 30_000, 300, 120


@pytest.fixture(scope="module")
def are():
    import torch
    assert torch.cuda.is_available()
    import paper_1308_2066_gb300 as are
    are.lib()
    return are


def elt(seed, nnz=5000):
    g = np.random.Generator(np.random.PCG64(seed))
    return g.permutation(CATALOG)[:nnz].astype(np.int32), g.lognormal(11, 1.5, nnz)


@pytest.mark.parametrize("nnz", [1500, 5000])     # bucketed in one launch, in two
@pytest.mark.parametrize("where", ["host", "device", "ids on the device"])
def test_memory_that_an_elt_takes(are, where, nnz):
    """Its entries and the offsets of its buckets, nothing beside them while it
    loads (the budget ends there); and with room for the entries alone, those."""
    import torch
    ids, losses = elt(1, nnz)
    a = torch.from_numpy(ids).cuda() if where != "host" else ids
    b = torch.from_numpy(losses).cuda() if where == "device" else losses
    entries, offsets = 12 * ids.size, 4 * (int(ids.max()) // 256 + 2)
    for room, takes in ((0, entries + offsets), (entries + offsets, entries + offsets),
                        (entries + offsets - 4, entries), (entries, entries)):
        ctx = are.are_create(0, room)
        try:
            are.are_load_elt(ctx, a, b)
            assert are.are_memory_used(ctx) == takes
        finally:
            are.are_destroy(ctx)
    ctx = are.are_create(0, entries - 4)
    try:
        with pytest.raises(are.AreError) as e:
            are.are_load_elt(ctx, a, b)
        assert e.value.status == are.ARE_ENOMEM and are.are_memory_used(ctx) == 0
        with pytest.raises(are.AreError) as e:                 # what is wrong with an ELT comes first
            are.are_load_elt(ctx, ids, -losses)
        assert e.value.status == are.ARE_EINVAL and are.are_memory_used(ctx) == 0
    finally:
        are.are_destroy(ctx)


def test_loading_from_the_host_waits_for_no_other_stream(are):
    import torch
    ids, losses = elt(2)
    ctx = are.are_create(0)
    try:
        are.are_free_elt(ctx, are.are_load_elt(ctx, ids, losses))   # its blocks are at hand from now on
        torch.cuda.synchronize()
        other = torch.cuda.Stream()
        with torch.cuda.stream(other):
            torch.cuda._sleep(400_000_000)                          # about 0.2 s
            done = torch.cuda.Event()
            done.record()
        are.are_load_elt(ctx, ids, losses)
        assert not done.query()
        done.synchronize()
    finally:
        are.are_destroy(ctx)


def test_elts_without_buckets(are):
    """Entries kept in the order given build the same rows; such a layer has no
    marks, in an analysis or on the server."""
    import torch
    elts = [elt(10 + j) for j in range(6)]
    ids = np.random.Generator(np.random.PCG64(3)).integers(0, CATALOG, N * K).astype(np.int32)
    spare = 1 << 22
    out = {}
    for bucketed in (True, False):
        room = 4 * (N * K + 64) + sum(12 * i.size for i, _ in elts) + spare
        ctx = are.are_create(0, room)
        try:
            y = are.are_load_yet(ctx, CATALOG, N, None, K, ids)
            hs = []
            for e in elts:
                if not bucketed:   # all but the entries' room taken while it loads
                    n = (room - are.are_memory_used(ctx) - 12 * e[0].size) // 4 - 64
                    held = are.are_load_yet(ctx, CATALOG, n, None, 1, np.zeros(n, np.int32))
                hs.append(are.are_load_elt(ctx, *e))
                if not bucketed:
                    are.are_free_yet(ctx, held)
            used = are.are_memory_used(ctx)
            layer = are.are_define_layer(ctx, hs, 3e4, 2e6, 0.0, INF)
            got = []
            for p in (0, 1):
                ylt = torch.full((N,), -1.0, dtype=torch.float64, device="cuda")
                are.are_simulate(ctx, layer, y, 0, N, p, ylt)
                got.append(ylt.cpu().numpy())
            marg = torch.zeros(N * K, dtype=torch.float64, device="cuda")
            are.are_simulate_occurrences(ctx, layer, y, 0, N, 0, marg, None, ylt)
            got += [marg.cpu().numpy(), ylt.cpu().numpy()]
            are.are_simulate_folded(ctx, layer, y, 0, N, ylt)
            got.append(ylt.cpu().numpy())
            are.are_free_layer(ctx, layer)
            assert are.are_memory_used(ctx) == used
            are.are_server_start(ctx, y, max_inflight=2, arena_bytes=1 << 21)
            r = are.are_wait(ctx, are.are_submit(ctx, hs, 3e4, 2e6, 0.0, INF, N, (20.0, 5.0), (0.9,)), 10_000_000)
            are.are_server_stop(ctx)
            pml, tvar = are.are_risk_measures(ctx, got[1], None, (20.0, 5.0), (0.9,))
            # FP32 losses, added by Kahan sums of either order
            np.testing.assert_allclose(r["pml"] + r["tvar"], np.concatenate([pml, tvar]), rtol=1e-6)
            out[bucketed] = got
        finally:
            are.are_destroy(ctx)
    assert (out[True][0] > 0).mean() > 0.2
    for a, b in zip(out[True], out[False]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("where", ["host", "device"])
@pytest.mark.parametrize("nnz", [1, 1023, 1025, 2047, 2048, 2049, 3000])
def test_every_entry_is_found(are, where, nnz):
    """One-event trials over the catalog give the losses back, whatever the
    order of the ids: sizes around a block's threads and its entries."""
    import torch
    ids, losses = elt(20 + nnz, nnz)
    want = np.zeros(CATALOG)
    want[ids] = losses
    if where == "device":
        ids, losses = torch.from_numpy(ids).cuda(), torch.from_numpy(losses).cuda()
    ctx = are.are_create(0)
    try:
        layer = are.are_define_layer(ctx, [are.are_load_elt(ctx, ids, losses)])
        y = are.are_load_yet(ctx, CATALOG, CATALOG, None, 1, np.arange(CATALOG, dtype=np.int32))
        out = torch.full((CATALOG,), -1.0, dtype=torch.float64, device="cuda")
        are.are_simulate(ctx, layer, y, 0, CATALOG, 0, out)
        np.testing.assert_array_equal(out.cpu().numpy(), want)
    finally:
        are.are_destroy(ctx)
