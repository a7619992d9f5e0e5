"""Accesses in critical sections, grouped by (location, lock) with a lock's sections in the order
of their acquires, against the oracle (which goes in trace order): sections of one lock whose
scopes do not overlap interleave access by access, sections nest, some are never released, and
one location is reached under many locks."""
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


def interleaved(seed, blocks, locks, locations, steps, nest, hold=False):
    """One agent per block; each step moves one agent on. Block-scope sections of all blocks run
    at the same time; now and then all of them end and a device-scope section follows."""
    rng = np.random.default_rng(seed)
    b = TG.TraceBuilder()
    held = [[] for _ in range(blocks)]

    def access(t):
        (b.wr if rng.random() < 0.4 else b.rd)(t, 0x40 + 8 * int(rng.integers(locations)))

    def drop(t, all_of_it=False):
        while held[t]:
            b.rel(t, held[t].pop(), TG.CTA)
            if not all_of_it:
                break

    for _ in range(steps):
        t = int(rng.integers(blocks))
        x = rng.random()
        free = [k for k in range(locks) if k not in held[t]]
        if x < 0.25 and len(held[t]) < nest and free:
            held[t].append(int(rng.choice(free)))
            b.acq(t, held[t][-1], TG.CTA)
        elif x < 0.4:
            drop(t)
        elif x < 0.44:
            for u in range(blocks):
                drop(u, True)
            k = int(rng.integers(locks))
            b.acq(t, k, TG.DEVICE)
            for _ in range(int(rng.integers(1, 4))):
                access(t)
            b.rel(t, k, TG.DEVICE)
        else:
            access(t)
    if not hold:
        for u in range(blocks):
            drop(u, True)
    return b.build(), TG.Geometry(blocks, 1, TG.WARP_GRAN)


@pytest.mark.parametrize("blocks,locks,locations,steps,nest,hold", [
    (1, 1, 1, 40, 1, True), (2, 1, 1, 60, 1, False), (5, 1, 2, 300, 1, True), (5, 3, 3, 600, 2, True),
    (40, 2, 4, 3000, 2, False), (40, 6, 1, 3000, 4, True), (70, 3, 5, 6000, 3, True), (3, 9, 200, 4000, 4, False)])
def test_interleaved_sections(gw, blocks, locks, locations, steps, nest, hold):
    ev, geo = interleaved(steps + blocks, blocks, locks, locations, steps, nest, hold)
    idx = np.nonzero(ev["op"] <= TG.REL)[0][:: max(1, len(ev) // 25)].tolist()
    want = O.run(ev, *geo.astuple(), clock_events=idx)
    with gw.Context(0) as c:
        c.set_clock_mode(gw.CLOCKS_DENSE)
        c.load_trace(ev, *geo.astuple())
        c.compute_order()
        assert np.array_equal(c.report_races(), want.races)
        for i in idx:
            assert np.array_equal(c.debug_clock(i, 0, geo.num_agents), want.clocks_c[i]), i
