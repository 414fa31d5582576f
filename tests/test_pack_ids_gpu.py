"""are_pack_ids around its blocks of 128 ids: the words against the bits laid
out one by one, and an id that does not fit anywhere in them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx_are():
    import paper_1308_2066_gb300 as are
    ctx = are.are_create(0)
    yield ctx, are
    are.are_destroy(ctx)


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 255, 256, 300])
def test_words_around_a_block(ctx_are, n):
    ctx, are = ctx_are
    g = np.random.default_rng(n)
    for bits in (1, 5, 8, 20, 21, 31, 32):
        ids = g.integers(0, min(1 << bits, 2**31 - 1), n).astype(np.int32)
        lay = ((ids[:, None].astype(np.uint64) >> np.arange(bits, dtype=np.uint64)) & np.uint64(1)).astype(np.uint8)
        lay = np.concatenate([lay.ravel(), np.zeros(-n * bits % 32, np.uint8)])
        want = np.packbits(lay, bitorder="little").view("<u4")
        out = np.full(want.size + 2, 0xABCDEF01, np.uint32)
        are.are_pack_ids(ctx, ids, bits, out)
        np.testing.assert_array_equal(out[:want.size], want)
        assert np.all(out[want.size:] == 0xABCDEF01)
        for at in {0, n // 2, n - 1}:
            for wrong in ([-1] if bits >= 31 else [-1, 1 << bits]):
                bad = ids.copy()
                bad[at] = wrong
                with pytest.raises(are.AreError) as e:
                    are.are_pack_ids(ctx, bad, bits, out)
                assert e.value.status == are.ARE_EINVAL and f"id {wrong} " in str(e.value)
