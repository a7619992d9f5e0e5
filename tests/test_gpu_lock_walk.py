"""The walk over a lock's sections (a warp per lock, batches of 32 entries) and the walk over an
agent's synchronisation entries (rounds of 32), against the oracle: entry counts around a batch,
few and many scopes per lock, device-scope acquires that join more scopes than a warp has lanes,
every nesting depth, and lists placed by a counter where their words exceed 32 bits."""
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


def check(gw, ev, geo):
    idx = np.nonzero(ev["op"] <= TG.REL)[0][:: max(1, len(ev) // 12)].tolist()
    want = O.run(ev, *geo.astuple(), clock_events=idx)
    with gw.Context(0) as c:
        c.set_clock_mode(gw.CLOCKS_DENSE)
        c.load_trace(ev, *geo.astuple())
        c.compute_order()
        assert np.array_equal(c.report_races(), want.races)
        for i in idx:
            assert np.array_equal(c.debug_clock(i, 0, geo.num_agents), want.clocks_c[i]), i


def sections(seed, blocks, apb, n, n_locks, p_dev, nest=1):
    """n sections, one after another (so none interleave), each up to `nest` locks deep."""
    rng = np.random.default_rng(seed)
    b = TG.TraceBuilder()
    for _ in range(n):
        t = int(rng.integers(blocks * apb))
        depth = int(rng.integers(1, nest + 1))
        locks = rng.choice(max(n_locks, depth), depth, replace=False).tolist()
        scopes = [TG.DEVICE if rng.random() < p_dev else TG.CTA for _ in locks]
        for lk, sc in zip(locks, scopes):
            b.acq(t, lk, sc)
            (b.wr if rng.random() < 0.3 else b.rd)(t, 0x100 + 8 * int(rng.integers(6)))
        for lk, sc in zip(reversed(locks), reversed(scopes)):
            b.rel(t, lk, sc)
        if rng.random() < 0.3:
            b.rd(int(rng.integers(blocks * apb)), 0x100 + 8 * int(rng.integers(6)))
    return b.build(), TG.Geometry(blocks * apb, apb, TG.WARP_GRAN)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 48, 200])
def test_batches(gw, n):
    check(gw, *sections(n, 3, 4, n, 1, 0.3))


@pytest.mark.parametrize("blocks,p_dev", [(1, 0.5), (40, 0.02), (63, 0.01), (64, 0.01), (150, 0.003), (319, 0.003),
                                          (40, 0.0), (40, 1.0)])
def test_scopes_of_a_lock(gw, blocks, p_dev):
    check(gw, *sections(blocks, blocks, 2, 6 * blocks + 100, 2, p_dev))


@pytest.mark.parametrize("nest", [1, 2, 3, 4])
def test_nesting(gw, nest):
    check(gw, *sections(nest, 4, 2, 150, 7, 0.4, nest))
    check(gw, *sections(10 + nest, 1, 1, 60, 5, 0.4, nest))


def test_lists_placed_by_a_counter(gw):
    # 2 * (320 scopes) words for each of 6.8M in-section accesses: more than 32 bits count
    blocks, per, n_sec = 319, 10_000, 680
    one = np.zeros(per + 2, dtype=TG.EVENT_DTYPE)
    one["op"] = TG.READ
    one["op"][0], one["op"][-1] = TG.ACQ, TG.REL
    one["scope"] = TG.CTA
    ev = np.tile(one, n_sec)
    sec = np.repeat(np.arange(n_sec), per + 2)
    ev["agent"] = sec * 7 % blocks
    ev["scope"][(ev["op"] >= TG.ACQ) & (sec % 5 == 0)] = TG.DEVICE
    ev["addr"] = np.where(ev["op"] >= TG.ACQ, 3, 0x1000 + 8 * ev["agent"].astype(np.uint64))
    ev["op"][1 : -1 : 50 * (per + 2)] = TG.WRITE
    ev["addr"][1 : -1 : 50 * (per + 2)] = 0x800
    ev = np.concatenate([ev, np.array([(2, TG.WRITE, 0, 0, 0, 0x800)], dtype=ev.dtype)])
    assert (len(ev) - 2 * n_sec) * 2 * (blocks + 1) > 2**32
    want = O.run(ev, blocks, 1, TG.WARP_GRAN)
    with gw.Context(0) as c:
        c.set_clock_mode(gw.CLOCKS_DENSE)
        c.load_trace(ev, blocks, 1, TG.WARP_GRAN)
        c.compute_order()
        races = c.report_races()
        assert np.array_equal(races, want.races)
    assert len(races)


def test_invalid_trace_comes_before_lack_of_memory(gw):
    # a section that interleaves with an overlapping one, under a limit that leaves no room for
    # the arrays after the lock walk
    ev, geo = sections(5, 8, 8, 4000, 3, 0.3)
    bad = np.concatenate([ev, np.array([(0, TG.ACQ, TG.DEVICE, 0, 0, 1), (9, TG.ACQ, TG.CTA, 0, 0, 1)], dtype=ev.dtype)])

    def result(events, limit):
        with gw.Context(0) as c:
            c.debug_alloc_limit(limit)
            c.load_trace(events, *geo.astuple())
            try:
                c.compute_order()
            except gw.GwcpError as e:
                return e.code, e.bad_index if e.code == gw.ERR_INVALID_TRACE else None
            return 0, None

    assert result(ev, 1 << 40)[0] == 0
    assert result(bad, 1 << 40) == (gw.ERR_INVALID_TRACE, len(ev) + 1)
    lo, hi = 0, 1 << 30  # the smallest limit that the valid trace fits
    while hi - lo > 1 << 12:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if result(ev, mid)[0] == 0 else (mid, hi)
    code = result(ev, lo)[0]
    assert code != 0 and code != gw.ERR_INVALID_TRACE
    assert result(bad, lo) == (gw.ERR_INVALID_TRACE, len(ev) + 1)
