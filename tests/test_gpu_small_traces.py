"""What a short trace is cut into, against the oracle: phase A's tiles and rounds with barriers
in them, the chunks of the allocation-free entry point's check (one location over many of
them), and the partner check's limit on the groups that a lane walks itself."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2111_12478_gb300 import tracegen as TG

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2111_12478_gb300 import gwcp

    return torch, gwcp


def races(gwcp, ev, geo):
    with gwcp.Context(0) as c:
        c.load_trace(ev, *geo.astuple())
        c.compute_order()
        return c.report_races()


def noalloc(env, ev, geo, cap):
    torch, gwcp = env
    dev = torch.from_numpy(ev.view(np.uint8).copy()).cuda()
    out = torch.zeros((max(cap, 1), 2), dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    rc, n, _ = gwcp.analyze_noalloc(dev.data_ptr(), len(ev), *geo.astuple(), out.data_ptr(), cap)
    assert rc == 0, gwcp.strerror(rc)
    return out.cpu().numpy().astype(np.uint64)[:n]


@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 255, 256, 257, 511, 513, 2047, 2049])
@pytest.mark.parametrize("blocks,apb,gran", [(8, 8, TG.WARP_GRAN), (1, 64, TG.THREAD), (40, 10, TG.WARP_GRAN),
                                             (70, 32, TG.WARP_GRAN)])
def test_tiles_and_barriers(env, n, blocks, apb, gran):
    ev, geo, _ = TG.generate(n, **dict(TG.WORKLOADS["8blk_64warp_10M"], n_events=n, num_blocks=blocks,
                                       agents_per_block=apb, granularity=gran, n_ranks=30, n_locks=5,
                                       p_barrier=0.15, p_syncwarp=0.5, p_acqrel=0.05))
    want = O.run(ev, *geo.astuple()).races
    assert np.array_equal(races(env[1], ev, geo), want)
    if geo.num_agents <= 256:
        assert np.array_equal(noalloc(env, ev, geo, len(want) + 4), want)


# one location over every chunk (chunks of 32 up to 131,072 accesses, then larger), with
# others at the trace's ends so that a chunk starts and ends inside a location
@pytest.mark.parametrize("n,W", [(30, 4), (32, 4), (33, 4), (64, 8), (1023, 8), (1057, 33), (3000, 200), (131_073, 8),
                                 (200_000, 3)])
def test_one_location_over_chunks(env, n, W):
    rng = np.random.default_rng(n)
    ev = np.zeros(n, dtype=TG.EVENT_DTYPE)
    ev["agent"] = rng.integers(W, size=n)
    ev["op"] = TG.ATOMIC  # device-scope updates never race with one another
    ev["scope"] = TG.DEVICE
    ev["addr"] = 0x100
    ev["addr"][rng.integers(n, size=max(1, n // 100))] = 0x80
    ev["addr"][rng.integers(n, size=max(1, n // 100))] = 0x180
    ev["op"][rng.integers(n, size=max(2, min(n // 20, 40)))] = TG.READ
    geo = TG.Geometry(W, 1, TG.WARP_GRAN)
    want = O.run(ev, *geo.astuple()).races
    assert np.array_equal(noalloc(env, ev, geo, len(want) + 4), want)


@pytest.mark.parametrize("W", [40, 48, 49, 50, 96, 97])
@pytest.mark.parametrize("ranked", [False, True])
def test_groups_around_the_limit(env, W, ranked):
    from paper_2111_12478_gb300 import ranker

    ev = np.zeros(W + 6, dtype=TG.EVENT_DTYPE)
    ev["agent"][:W] = np.random.default_rng(W).permutation(W)
    ev["agent"][W:] = np.arange(6) % 3
    ev["op"][W:] = TG.WRITE
    ev["addr"] = 0x100
    geo = TG.Geometry(W, 1, TG.WARP_GRAN)
    want = O.run(ev, *geo.astuple()).races
    with env[1].Context(0) as c:
        if ranked:
            c.set_ranker(ranker.init_theta(2))
        c.load_trace(ev, *geo.astuple())
        c.compute_order()
        assert np.array_equal(c.report_races(), want)
    assert len(want)
