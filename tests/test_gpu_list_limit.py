"""The partner check's limit on the groups a lane walks itself, which follows from how many
accesses of the trace have more: counts of such accesses around the most that are put aside, at
list lengths around the first steps, against the oracle."""
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


def long_lists(W, updates, seed):
    """All but three of W agents (two blocks) read one location and meet at their block's barrier;
    then `updates` device-scope updates, each with the W - 3 reading agents' groups."""
    rng = np.random.default_rng(seed)
    n = W - 3
    ev = np.zeros(n + 2 + updates, dtype=TG.EVENT_DTYPE)
    ev["addr"] = 0x40
    ev["agent"][:n] = rng.permutation(n)
    ev["op"][n:n + 2], ev["scope"][n:n + 2], ev["addr"][n:n + 2] = TG.BARRIER, TG.CTA, [0, 1]
    ev["agent"][n:n + 2] = [0, W // 2]
    ev["agent"][n + 2:] = rng.integers(0, W, updates)
    ev["op"][n + 2:], ev["scope"][n + 2:] = TG.ATOMIC, TG.DEVICE
    return ev, (W, W // 2, TG.WARP_GRAN)


@pytest.mark.parametrize("W", [34, 36, 52, 100])
@pytest.mark.parametrize("updates", [300, 8191, 8192, 8193])
@pytest.mark.parametrize("ranked", [False, True])
def test_counts_around_the_most_put_aside(gw, W, updates, ranked):
    from paper_2111_12478_gb300 import ranker

    ev, geo = long_lists(W, updates, W + updates)
    want = O.run(ev, *geo).races
    assert len(want) > updates
    with gw.Context(0) as c:
        if ranked:
            c.set_ranker(ranker.init_theta(2))
        for _ in range(2):
            c.load_trace(ev, *geo)
            c.compute_order()
            assert np.array_equal(c.report_races(), want)
