"""Short traces of barriers over many agents, against the oracle: a barrier has an entry per
member, so the synchronisation entries outnumber the events by up to 1024 to 1 and the scratch
of the scans over them cannot be sized by the events."""
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


def barriers(apb, n, seed):
    """One block: n events, a CTA barrier each but for the writes and reads of a few locations."""
    rng = np.random.default_rng(seed)
    ev = np.zeros(n, dtype=TG.EVENT_DTYPE)
    ev["agent"] = rng.integers(0, apb, n)
    ev["op"], ev["scope"] = TG.BARRIER, TG.CTA
    at = rng.random(n) < 0.3
    ev["op"][at] = rng.choice([TG.READ, TG.WRITE], at.sum())
    ev["scope"][at] = 0
    ev["addr"][at] = 4 * rng.integers(0, 3, at.sum())
    return ev, (apb, apb, TG.THREAD)


@pytest.mark.parametrize("apb,n", [(1024, 40), (1024, 1300), (512, 2600)])
def test_barrier_entries(gw, apb, n):
    ev, geo = barriers(apb, n, n)
    want = O.run(ev, *geo).races
    with gw.Context(0) as c:
        for _ in range(2):
            c.load_trace(ev, *geo)
            c.compute_order()
            assert np.array_equal(c.report_races(), want)
