"""The tile walker against the oracle: widths and block sizes from one tile to sixteen, blocks
of one walker (nobody helps with a merge) to 32, many sections per barrier period (more
posted merges than places), barriers between them; and 512 agents dense, as tiles, and as
tiles after a dense analysis has run out of memory."""
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


def heavy(seed, blocks, apb, n, **kw):
    p = dict(TG.WORKLOADS["8blk_64warp_10M"], n_events=n, num_blocks=blocks, agents_per_block=apb, n_ranks=60,
             n_locks=40, p_acqrel=0.1, p_barrier=0.05, nest_prob=0.3, cs_len_mean=2.0, plant_frac=0.02)
    p.update(kw)
    ev, geo, _ = TG.generate(seed, **p)
    return ev, geo.astuple()


def check(gw, ev, geo, mode, clocks=6, **kw):
    pick = np.nonzero(ev["op"] <= TG.REL)[0]
    idx = pick[:: max(1, len(pick) // clocks)].tolist() if clocks else []
    want = O.run(ev, *geo, clock_events=idx, **kw)
    with gw.Context(0, **kw) as c:
        c.set_clock_mode(mode)
        for _ in range(2):
            c.load_trace(ev, *geo)
            c.compute_order()
            assert np.array_equal(c.report_races(), want.races)
        for i in idx:
            assert np.array_equal(c.debug_clock(i, 0, geo[0]), want.clocks_c[i]), i


@pytest.mark.parametrize("blocks,apb", [(8, 1), (30, 7), (8, 32), (64, 8), (16, 32), (40, 31), (300, 4), (128, 32)])
def test_shapes(gw, blocks, apb):
    check(gw, *heavy(blocks + apb, blocks, apb, 8000), gw.CLOCKS_TILES)


@pytest.mark.parametrize("p_barrier", [0.0, 0.3])
def test_many_sections(gw, p_barrier):
    check(gw, *heavy(5, 20, 32, 12000, p_acqrel=0.5, n_locks=200, p_barrier=p_barrier), gw.CLOCKS_TILES)


@pytest.mark.parametrize("kw", [dict(hb_only=True), dict(forced_barrier=True)])
def test_variants(gw, kw):
    check(gw, *heavy(9, 24, 32, 8000), gw.CLOCKS_TILES, clocks=0, **kw)


@pytest.mark.parametrize("blocks,apb", [(64, 8), (32, 16), (16, 32), (12, 24), (15, 20), (75, 8)])
def test_automatic_choice(gw, blocks, apb):
    check(gw, *heavy(blocks, blocks, apb, 6000), gw.CLOCKS_AUTO)


def test_512_agents_fall_back_to_tiles(gw):
    # many sections: three dense clocks of 2 KB each are published per release
    ev, geo = heavy(3, 64, 8, 300_000, p_acqrel=0.8, p_barrier=0.0, n_locks=4000, n_ranks=40_000, plant_frac=0.001)
    want = O.run(ev, *geo).races
    used = {}
    for mode in (gw.CLOCKS_DENSE, gw.CLOCKS_TILES):
        with gw.Context(0) as c:
            c.set_clock_mode(mode)
            c.load_trace(ev, *geo)
            c.compute_order()
            used[mode] = c.clock_bytes()["reserved"]


    def analyse(mode, limit):  # the clock versions' bytes, or None when out of memory
        with gw.Context(0) as c:
            c.set_clock_mode(mode)
            c.debug_alloc_limit(limit)
            c.load_trace(ev, *geo)
            try:
                c.compute_order()
            except gw.GwcpError as e:
                assert e.code == gw.ERR_OOM
                return None
            c.debug_alloc_limit(0)  # (the copy of the races needs a buffer too)
            assert np.array_equal(c.report_races(), want)
            return c.clock_bytes()["reserved"]

    least = {}
    for mode in used:  # the smallest limit that is enough, to 1 MB
        lo, hi = 1 << 20, 1 << 30
        while hi - lo > 1 << 20:
            mid = (lo + hi) // 2
            lo, hi = (lo, mid) if analyse(mode, mid) else (mid, hi)
        least[mode] = hi
    assert least[gw.CLOCKS_TILES] + (4 << 20) < least[gw.CLOCKS_DENSE]
    assert analyse(gw.CLOCKS_AUTO, least[gw.CLOCKS_DENSE]) == used[gw.CLOCKS_DENSE]
    # (the number of tiles handed out varies a little with the walkers' timing)
    for limit in (least[gw.CLOCKS_DENSE] - (2 << 20), least[gw.CLOCKS_TILES] + (1 << 20)):
        got = analyse(gw.CLOCKS_AUTO, limit)
        assert got and got != used[gw.CLOCKS_DENSE]
    assert analyse(gw.CLOCKS_AUTO, least[gw.CLOCKS_TILES] - (2 << 20)) is None
