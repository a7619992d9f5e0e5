"""The automatic choice between dense clocks and tiles: what fits device memory one way is
analysed that way when the choice does not fit, and with the chunked check the choice is dense
below 512 agents and tiles from there, whenever the check mode is set."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2111_12478_gb300 import tracegen as TG

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


def trace(blocks, apb, n=6000):
    ev, geo, _ = TG.generate(blocks, **dict(TG.WORKLOADS["8blk_64warp_10M"], n_events=n, num_blocks=blocks,
                                            agents_per_block=apb, n_ranks=200, n_locks=20, p_acqrel=0.05))
    return ev, geo.astuple()


@pytest.mark.parametrize("blocks,apb", [(16, 24), (9, 32), (30, 17)])
def test_dense_where_tiles_do_not_fit(gw, blocks, apb):
    ev, geo = trace(blocks, apb)
    want = O.run(ev, *geo).races

    def fits(mode, limit):
        with gw.Context(0) as c:
            c.set_clock_mode(mode)
            c.debug_alloc_limit(limit)
            for _ in range(2):
                c.load_trace(ev, *geo)
                try:
                    c.compute_order()
                except gw.GwcpError as e:
                    assert e.code == gw.ERR_OOM
                    return False
            c.debug_alloc_limit(0)  # (the copy of the races needs a buffer too)
            assert np.array_equal(c.report_races(), want)
            return True

    lo, hi = 1 << 20, 1 << 28
    while hi - lo > 1 << 20:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(gw.CLOCKS_DENSE, mid) else (mid, hi)
    assert not fits(gw.CLOCKS_TILES, hi)
    assert fits(gw.CLOCKS_AUTO, hi) and not fits(gw.CLOCKS_AUTO, lo - (1 << 20))


@pytest.mark.parametrize("blocks,apb,tiles", [(16, 24, False), (16, 31, False), (64, 8, True), (16, 32, True)])
@pytest.mark.parametrize("late", [False, True])
def test_choice_with_the_chunked_check(gw, blocks, apb, tiles, late):
    ev, geo = trace(blocks, apb)
    want = O.run(ev, *geo).races
    with gw.Context(0) as c:
        if not late:
            c.set_check_mode(gw.CHECK_CHUNKED)
        c.load_trace(ev, *geo)
        if late:
            c.set_check_mode(gw.CHECK_CHUNKED)
        c.compute_order()
        assert np.array_equal(c.report_races(), want)
        b = c.clock_bytes()
        assert (b["stored"] != b["dense"]) == tiles
        c.set_check_mode(gw.CHECK_AUTO)
        c.compute_order()
        assert np.array_equal(c.report_races(), want)
        b = c.clock_bytes()
        assert (b["stored"] != b["dense"]) == (apb > 16)
