"""The radix sort when its tiles give up waiting for the tiles before them: with a limit of no
looks at all (most tiles then count for themselves), a few, and the usual one, the result is the
stable sort. Sizes of one block, both tile sizes and their remainders; masks with scattered
bits, adjacent ones and none of a digit's share."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2111_12478_gb300 import gwcp

    return gwcp


@pytest.mark.parametrize("polls", [0, 3, 1 << 22])
@pytest.mark.parametrize("n,mask,with_vals", [
    (1, 0xFF, True), (4096, 0x0F0F0F, True), (4097, 0xFFFF, True), (5000, 0xFFFFFFFFFFFFFFFF, False),
    (1 << 18, 0x1111111111, True), ((1 << 18) + 1, 0xFFF, True), (1_000_003, 0x8000_0000_0FFF_8001, True),
    (2_500_000, 0x000F_FFFF_0003_FFFF, False)])
def test_sort(gw, n, mask, with_vals, polls):
    rng = np.random.default_rng(n)
    # few distinct digits in one half: long runs of equal keys, whose order must stay
    keys = rng.integers(0, 1 << 63, n, dtype=np.uint64) * np.uint64(2) + rng.integers(0, 2, n, dtype=np.uint64)
    keys[::2] &= np.uint64(0x0300_0000_0000_0301)
    order = np.argsort(keys & np.uint64(mask), kind="stable")
    vals = np.arange(n, dtype=np.uint32) if with_vals else None
    got = keys.copy()
    gw.debug_sort(0, got, vals, mask, polls)
    assert np.array_equal(got, keys[order])
    if with_vals:
        assert np.array_equal(vals, order.astype(np.uint32))
