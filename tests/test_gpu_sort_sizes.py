"""The sorts and scans of an analysis at the sizes where they change form (one block, tiles of
1,024 and of 3,072 pairs; one block, two and three kernels), against the oracle: traces whose
access, lock and race counts lie at those edges, keys with few and with scattered varying bits."""
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


def run(gw, ev, geo, **kw):
    with gw.Context(0) as c:
        if kw.get("check") is not None:
            c.set_check_mode(kw["check"])
        c.load_trace(ev, *geo)
        c.compute_order()
        return c.report_races()


def accesses(n, seed, spread, agents=64):
    """n accesses without synchronisation; `spread` scatters the address bits that vary."""
    rng = np.random.default_rng(seed)
    ev = np.zeros(n, dtype=TG.EVENT_DTYPE)
    ev["agent"] = rng.integers(agents, size=n)
    loc = rng.integers(max(2, n // 3), size=n).astype(np.uint64)
    addr = np.zeros(n, dtype=np.uint64)
    for b in range(20):
        addr |= ((loc >> np.uint64(b)) & np.uint64(1)) << np.uint64(2 + b * spread)
    ev["addr"] = addr
    ev["op"] = np.where(rng.random(n) < 0.1, TG.WRITE, TG.READ)
    return ev, (agents, 8, TG.WARP_GRAN)


@pytest.mark.parametrize("n", [2, 1023, 4095, 4096, 4097, 5119, 5120, 16384, 16385, 65537, 262143, 262144, 262145, 300001])
@pytest.mark.parametrize("spread", [1, 2])
def test_access_counts(gw, n, spread):
    ev, geo = accesses(n, n, spread)
    want = O.run(ev, *geo).races
    for check in (gw.CHECK_SPARSE, gw.CHECK_CHUNKED):
        assert np.array_equal(run(gw, ev, geo, check=check), want)


def test_one_location_and_one_agent(gw):
    ev, geo = accesses(20_000, 1, 1)
    ev["addr"] = 0x40
    ev["op"][100:] = TG.READ
    assert np.array_equal(run(gw, ev, geo), O.run(ev, *geo).races)
    ev["agent"] = 3
    assert len(run(gw, ev, geo)) == 0


@pytest.mark.parametrize("n", [40_000, 120_000])
def test_many_locks_and_barriers(gw, n):
    p = dict(TG.WORKLOADS["8blk_64warp_10M"], n_events=n, n_ranks=500, n_locks=3000, p_acqrel=0.5, p_barrier=0.02)
    ev, geo, _ = TG.generate(5, **p)
    geo = geo.astuple()
    assert np.array_equal(run(gw, ev, geo), O.run(ev, *geo).races)
