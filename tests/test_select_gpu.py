"""PML and TVaR of one YLT and of several at a time, where the selection can go
wrong: one value, sizes around a block's share, long runs of ties with other
values in their bin, more distinct keys in a bin than are kept (the radix
passes), values of both signs, targets that share a bin, and more YLTs than
are selected at a time.  The order statistics are bit-exact; a mean is a sum of
m values, rounded once, against math.fsum: one rounding of the sum and one of
the quotient."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RPS = [1.0, 2.0, 3.0, 10.0, 100.0, 250.0]
LEVELS = [0.5, 0.99]


@pytest.fixture(scope="module")
def are():
    import torch
    assert torch.cuda.is_available()
    import paper_1308_2066_gb300 as are
    are.lib()
    return are


@pytest.fixture(scope="module")
def ctx(are):
    c = are.are_create(0)
    yield c
    are.are_destroy(c)


def draw(kind, n, g):
    y = g.lognormal(14, 2.0, n)
    if kind == "ties":             # a cap held by many, with other values just above and below it
        y[g.random(n) < 0.3] = 1e8
        y[g.random(n) < 0.2] = 0.0
        near = g.random(n) < 0.01
        y[near] = 1e8 * (1.0 + 1e-6 * g.normal(size=int(near.sum())))
    elif kind == "narrow":         # every key in one or two bins
        y = 1e6 * (1.0 + 1e-7 * g.random(n))
    elif kind == "signed":
        y = g.normal(size=n) * 10.0 ** g.integers(-3, 9, n)
        y[g.random(n) < 0.1] = -0.0
    elif kind == "constant":
        y[:] = 7.25
    return y


def expected(y, orc):
    s = np.sort(y)[::-1]
    n = y.size
    return (np.array([s[orc.rank_for_return_period(n, r) - 1] for r in RPS]),
            np.array([math.fsum(s[: orc.rank_for_level(n, a)]) / orc.rank_for_level(n, a) for a in LEVELS]))


@pytest.mark.parametrize("kind", ["plain", "ties", "narrow", "signed", "constant"])
@pytest.mark.parametrize("n", [1, 2, 1023, 8192, 8193, 100_003, 1_000_000])
def test_one_ylt(are, ctx, orc, kind, n):
    import torch
    y = draw(kind, n, np.random.default_rng(n))
    want_pml, want_tv = expected(y, orc)
    d = torch.from_numpy(y).cuda()
    out = (torch.full((len(RPS),), -1.0, dtype=torch.float64, device="cuda"),
           torch.full((len(LEVELS),), -1.0, dtype=torch.float64, device="cuda"))
    for rps, lv in ((RPS, LEVELS), (RPS[:1], []), ([], LEVELS)):    # again on the same scratch
        pml, tv = are.are_risk_measures(ctx, d, n, rps, lv)
        np.testing.assert_array_equal(pml, want_pml[: len(rps)])
        np.testing.assert_allclose(tv, want_tv[: len(lv)], rtol=2.0 ** -51)
    are.are_risk_measures(ctx, d, n, RPS, LEVELS, out=out)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out[0].cpu().numpy(), want_pml)
    np.testing.assert_allclose(out[1].cpu().numpy(), want_tv, rtol=2.0 ** -51)


@pytest.mark.parametrize("n_ylt,n", [(1, 5000), (3, 200_001), (17, 20_000), (40, 3000)])
def test_many_ylts(are, ctx, orc, n_ylt, n):
    import torch
    g = np.random.default_rng(n_ylt)
    kinds = ["plain", "ties", "signed", "constant"] + (["narrow"] if n_ylt != 17 else [])
    ys = [draw(kinds[i % len(kinds)], n, g) for i in range(n_ylt)]
    d = [torch.from_numpy(y).cuda() for y in ys]
    for _ in range(2):
        pml, tv = are.are_risk_measures_batch(ctx, d, n, RPS, LEVELS)
        for i, y in enumerate(ys):
            want_pml, want_tv = expected(y, orc)
            np.testing.assert_array_equal(pml[i], want_pml)
            np.testing.assert_allclose(tv[i], want_tv, rtol=2.0 ** -51, atol=1e-300)
