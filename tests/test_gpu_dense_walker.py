"""The walker with clocks in registers against the oracle, over its shapes: widths and block
sizes (barriers joined in shared memory or in global memory, every choice of staging that the
shared memory leaves), plans shorter and longer than a batch of 16 entries, releases with more
records than a warp has lanes, acquires that join more than four releases, warp barriers."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2111_12478_gb300 import tracegen as TG
from paper_2111_12478_gb300.tracegen import THREAD, WARP_GRAN

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


def check(gw, ev, geo, clocks=8, mode=None, **kw):
    idx = []
    if clocks:
        pick = np.nonzero(ev["op"] <= TG.REL)[0]
        idx = pick[:: max(1, len(pick) // clocks)].tolist()
    okw = {k: v for k, v in kw.items()}
    want = O.run(ev, *geo.astuple(), clock_events=idx, **okw)
    with gw.Context(0, **kw) as c:
        c.set_clock_mode(gw.CLOCKS_DENSE if mode is None else mode)
        c.load_trace(ev, *geo.astuple())
        c.compute_order()
        assert np.array_equal(c.report_races(), want.races)
        for i in idx:
            assert np.array_equal(c.debug_clock(i, 0, geo.num_agents), want.clocks_c[i]), i


def heavy(seed, blocks, apb, gran, n, **kw):
    p = dict(TG.WORKLOADS["8blk_64warp_10M"], n_events=n, num_blocks=blocks, agents_per_block=apb, granularity=gran,
             n_ranks=60, n_locks=24, p_acqrel=0.06, p_barrier=0.1, p_syncwarp=0.5, nest_prob=0.3,
             cs_len_mean=2.0, plant_frac=0.02)
    p.update(kw)
    ev, geo, _ = TG.generate(seed, **p)
    return ev, geo


SHAPES = [(8, 8, WARP_GRAN), (2, 2, WARP_GRAN), (5, 7, WARP_GRAN), (32, 8, WARP_GRAN), (8, 32, WARP_GRAN),
          (16, 32, WARP_GRAN), (64, 16, WARP_GRAN), (32, 32, WARP_GRAN), (100, 1, WARP_GRAN), (1, 32, THREAD),
          (4, 24, THREAD), (1, 64, THREAD), (3, 50, THREAD), (2, 256, THREAD), (1, 1000, THREAD)]


@pytest.mark.parametrize("blocks,apb,gran", SHAPES)
def test_shapes(gw, blocks, apb, gran):
    check(gw, *heavy(blocks + apb, blocks, apb, gran, 6000))


@pytest.mark.parametrize("n", [3, 40, 150, 300, 1200])
def test_short_plans(gw, n):
    check(gw, *heavy(n, 4, 8, WARP_GRAN, n, p_acqrel=0.4, p_barrier=0.05))


def test_many_records_per_release(gw):
    # two locks, many sections each: a release meets more than 32 records
    check(gw, *heavy(3, 8, 8, WARP_GRAN, 20000, n_locks=2, p_barrier=0.0002))


def test_acquire_joins_many_scopes(gw):
    # block-scoped sections of one lock in many blocks, then a device-scoped one joins them all
    b = TG.TraceBuilder()
    for r in range(3):
        for blk in range(12):
            t = blk * 4 + r
            b.acq(t, 0, TG.CTA)
            b.wr(t, 0x100)
            b.rel(t, 0, TG.CTA)
        b.acq(r, 0, TG.DEVICE)
        b.rd(r, 0x100)
        b.wr(r, 0x100)
        b.rel(r, 0, TG.DEVICE)
    for t in range(48):
        b.rd(t, 0x100)
    check(gw, b.build(), TG.Geometry(48, 4, WARP_GRAN), clocks=40)


@pytest.mark.parametrize("kw", [dict(hb_only=True), dict(forced_barrier=True)])
def test_variants(gw, kw):
    check(gw, *heavy(11, 8, 8, WARP_GRAN, 6000), clocks=0, **kw)
    check(gw, *heavy(12, 2, 96, THREAD, 6000), clocks=0, **kw)


@pytest.mark.parametrize("blocks,apb,gran", [(8, 8, WARP_GRAN), (32, 8, WARP_GRAN), (3, 50, THREAD), (32, 32, WARP_GRAN)])
def test_compressed(gw, blocks, apb, gran):
    check(gw, *heavy(blocks, blocks, apb, gran, 5000), clocks=0, mode=gw.CLOCKS_COMPRESSED)
