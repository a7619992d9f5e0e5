"""The partner check at locations that many agents touched, against the oracle: an access
with more than 192 partner groups is cut by agent and shared by the lanes of warps (items of
a second kernel, or with a ranker the lanes of its own warp)."""
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


def hot_trace(W, apb, writes, classes=1, seed=0):
    """Every agent reads one location (in a random order; some also write it or update it
    atomically at either scope when classes > 1), then `writes` writes by a few agents."""
    rng = np.random.default_rng(seed)
    rows = []
    for c in range(classes):
        for t in rng.permutation(W):
            op, scope = ((TG.READ, 0), (TG.WRITE, 0), (TG.ATOMIC, TG.CTA), (TG.ATOMIC, TG.DEVICE))[c]
            if c == 0 or rng.random() < 0.9:
                rows.append((t, op, scope, 0, 0, 0x1000))
            if rng.random() < 0.05:
                rows.append((t, TG.BARRIER, TG.CTA, 0, 0, t // apb))
    for k in range(writes):
        rows.append((int(rng.integers(min(W, 5))), TG.WRITE if k % 3 else TG.READ, 0, 0, 0, 0x1000))
    ev = np.zeros(len(rows), dtype=TG.EVENT_DTYPE)
    for i, r in enumerate(rows):
        ev[i] = r
    return ev, TG.Geometry(W, apb, TG.WARP_GRAN)


# group counts around the limit (192), one to four class lists, clocks dense and as tiles
CASES = [(184, 8, 3, 1), (192, 8, 3, 1), (200, 8, 3, 1), (64, 8, 7, 4), (96, 8, 5, 3), (320, 8, 9, 2), (512, 8, 4, 4),
         (1024, 32, 3, 1), (1088, 32, 40, 2)]


@pytest.mark.parametrize("W,apb,writes,classes", CASES)
@pytest.mark.parametrize("ranked", [False, True])
def test_many_partner_groups(gw, W, apb, writes, classes, ranked):
    from paper_2111_12478_gb300 import ranker

    ev, geo = hot_trace(W, apb, writes, classes, seed=W + classes)
    want = O.run(ev, *geo.astuple()).races
    with gw.Context(0, timeline=True) as c:
        if ranked:
            c.set_ranker(ranker.init_theta(2))
        c.load_trace(ev, *geo.astuple())
        c.compute_order()
        got = c.report_races()
        _, _, per = c.check_timeline()
    assert len(want) > 0 and np.array_equal(got, want)
    assert int(per.sum()) == len(want)


def test_compressed_versions(gw):
    ev, geo = hot_trace(256, 8, 6, 4, seed=1)
    want = O.run(ev, *geo.astuple()).races
    with gw.Context(0) as c:
        c.set_clock_mode(gw.CLOCKS_COMPRESSED)
        c.load_trace(ev, *geo.astuple())
        c.compute_order()
        assert np.array_equal(c.report_races(), want)


def test_more_items_than_room(gw):
    # 3400 accesses of at least 32 items each: over n / 8 + 65536 items
    ev, geo = hot_trace(4096, 32, 3400)
    want = O.run(ev, *geo.astuple()).races
    with gw.Context(0) as c:
        for _ in range(2):
            c.load_trace(ev, *geo.astuple())
            c.compute_order()
            assert np.array_equal(c.report_races(), want)
