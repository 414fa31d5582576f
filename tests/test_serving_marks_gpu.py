"""The pricing server's requests over marked events: arenas that hold their
marks, and arenas that do not."""
import math

import numpy as np
import pytest

import workloads as W
from gpu_support import rel_close

pytestmark = pytest.mark.gpu
INF = math.inf
N_TRIALS, K, CATALOG = 3000, 100, 20_000
RPS, LEVELS = (100.0, 20.0), (0.99,)


@pytest.fixture(scope="module")
def are():
    import torch
    assert torch.cuda.is_available()
    import paper_1308_2066_gb300 as are
    are.lib()
    return are


def up(n):
    """The arena hands out blocks of whole 256 bytes."""
    return (n + 255) // 256 * 256


# dense rows of 32 and 64 bytes, read by the persistent kernel without marks
@pytest.mark.parametrize("J", [6, 12])
def test_arenas_around_the_size_that_holds_the_marks(are, orc, J):
    """A request is served in an arena that holds its table and its trial
    losses, whether or not the marks fit beside them; with their blocks rounded
    up, they may just not."""
    g = np.random.Generator(np.random.PCG64(61 + J))
    yet = W.yet_fixed(g, N_TRIALS, K, CATALOG, timestamps=False)
    elts = [W.elt_lognormal(g, CATALOG, 400) for _ in range(J)]
    wl = W.Workload("s", yet, elts, [W.Layer(list(range(J)), 5e4, 2e6, 1e5, INF)])
    pml, tvar = orc.risk_measures(orc.simulate_layer(wl).ylt, RPS, LEVELS)
    rows, marks, ylt = CATALOG * (32 if J <= 8 else 64), (CATALOG + 127) // 128 * 16, 8 * N_TRIALS
    assert marks % 256 and rows % 256 == 0
    ctx = are.are_create(0)
    try:
        y = are.are_load_yet(ctx, CATALOG, N_TRIALS, None, K, yet.ids)
        hs = [are.are_load_elt(ctx, e.ids, e.losses, e.fx, e.ded, e.lim, e.share) for e in elts]
        whole = rows + up(marks) + up(ylt)
        for arena in (rows + up(ylt), rows + marks + up(ylt) - 1, rows + marks + up(ylt), whole - 1, whole, 2 * whole):
            are.are_server_start(ctx, y, max_inflight=2, arena_bytes=arena)
            tickets = [are.are_submit(ctx, hs, 5e4, 2e6, 1e5, INF, N_TRIALS, RPS, LEVELS) for _ in range(2)]
            for t in tickets:
                r = are.are_wait(ctx, t, 10_000_000)
                assert r["status"] == are.ARE_OK, (arena, r)
                assert rel_close(r["pml"], pml, 1e-5) and rel_close(r["tvar"], tvar, 1e-5), (arena, r)
            are.are_server_stop(ctx)
    finally:
        are.are_destroy(ctx)
