"""What an analysis that failed leaves behind in its context: nothing that the next trace pays
for."""
import numpy as np
import pytest

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


def overlapping_sections(agents, apb):
    """Two agents in one device-scoped lock at once: found by the lock walk only."""
    ev = np.zeros(4, dtype=TG.EVENT_DTYPE)
    ev["agent"], ev["op"], ev["scope"], ev["addr"] = [0, 1, 1, 0], [TG.ACQ, TG.ACQ, TG.REL, TG.REL], TG.DEVICE, 7
    return ev, (agents, apb, TG.WARP_GRAN)


def launches(gw, c, ev, geo):
    before = gw.launch_count()
    c.load_trace(ev, *geo)
    c.compute_order()
    races = c.report_races()
    return gw.launch_count() - before, races


@pytest.mark.parametrize("mode", ["CLOCKS_COMPRESSED", "CLOCKS_DENSE", "CLOCKS_TILES"])
def test_trace_after_an_invalid_one(gw, mode):
    ev, geo, _ = TG.generate(3, workload="8blk_64warp_10M", n_events=200_000)
    geo = geo.astuple()
    with gw.Context(0) as c:
        c.set_clock_mode(getattr(gw, mode))
        want, races = launches(gw, c, ev, geo)
    with gw.Context(0) as c:
        c.set_clock_mode(getattr(gw, mode))
        bad, bgeo = overlapping_sections(*geo[:2])
        c.load_trace(bad, *bgeo)
        with pytest.raises(gw.GwcpError) as e:
            c.compute_order()
        assert e.value.code == gw.ERR_INVALID_TRACE and e.value.bad_index == 1
        got, again = launches(gw, c, ev, geo)
        assert got <= want  # (one pass over the trace, as in a new context)
        assert np.array_equal(again, races)


def test_long_invalid_trace_ends_at_the_lock_walk(gw):
    def failing(n):
        ev = np.zeros(n + 4, dtype=TG.EVENT_DTYPE)
        rng = np.random.default_rng(n)
        ev["agent"], ev["addr"] = rng.integers(0, 64, n + 4), 4 * rng.integers(0, 1000, n + 4)
        ev["op"] = rng.choice([TG.READ, TG.WRITE], n + 4)
        bad, geo = overlapping_sections(64, 8)
        ev[n:] = bad
        return ev, geo

    taken = {}
    for n in (100_000, 1 << 23):
        ev, geo = failing(n)
        with gw.Context(0) as c:
            before = gw.launch_count()
            c.load_trace(ev, *geo)
            with pytest.raises(gw.GwcpError) as e:
                c.compute_order()
            taken[n] = gw.launch_count() - before
        assert e.value.code == gw.ERR_INVALID_TRACE and e.value.bad_index == n + 1
    assert taken[1 << 23] < taken[100_000]  # no sort, grouping or check behind the lock walk
