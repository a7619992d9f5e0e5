"""The analyses that this library is run for, as measurable cases.

A case is one trace (or one batch of traces, or one set of ranker rows) and the options a
caller gives; ``prepare`` holds what the caller has in hand, ``run`` makes one pass through
the public entry points and returns the results whole.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2111_12478_gb300 import gwcp, ranker, tracegen

MIX64 = tracegen.WORKLOADS["8blk_64warp_10M"]
MIX8192 = tracegen.WORKLOADS["256blk_8192warp_200M"]
MIXTHREAD = tracegen.WORKLOADS["tiny_1blk_64thr_10k"]

# races per event of the mixes' traces, for the bytes a pass has to write (the counts of
# the generated traces; they grow with the width because a planted access meets more agents)
RACES_64, RACES_WIDE, RACES_8192, RACES_THREAD = 0.1, 0.5, 0.0001, 0.05


def listed():
    return [
        # the smallest trace of the benchmark: one block of 64 threads, thread granularity,
        # block- and warp-scope barriers; a debugging run on one kernel of a test suite
        dict(name="tiny_64thr_10k", kind="trace", mix="thread", blocks=1, apb=64, n=10_000),
        # the allocation-free entry point of a runtime hook: a small trace, races left on the device
        dict(name="hook_64warp_60k", kind="noalloc", blocks=8, apb=8, n=60_001),
        # several blocks at thread granularity (a block is wider than a walker CTA's 32 agents,
        # so barriers go through global memory)
        dict(name="thread_256thr_250k", kind="trace", mix="thread", blocks=2, apb=128, n=250_007),
        # the 8-block, 64-warp benchmark trace, resident on the device
        dict(name="warp64_10M", kind="trace", mix="64", blocks=8, apb=8, n=10_000_000),
        # a middle width, from pinned host memory: copy in, analysis, races out
        dict(name="host_256warp_5M", kind="trace", mix="64", blocks=32, apb=8, n=5_000_001, host=True),
        # the first width kept as tile tables
        dict(name="warp512_2M", kind="trace", mix="64", blocks=64, apb=8, n=2_345_679),
        # a wide trace of the batched and served workloads (blocks of 32 warps)
        dict(name="warp4096_4M", kind="trace", mix="64", blocks=128, apb=32, n=4_000_000),
        # the 256-block, 8192-warp benchmark trace, its first 50M events (the prefix whose races
        # are stored with the tests); the largest case
        dict(name="warp8192_50M", kind="trace", mix="8192", blocks=256, apb=32, n=50_000_000),
        # the paper's memory mode: compressed clock versions with forced barrier compression
        dict(name="memory_64warp_3M", kind="trace", mix="64", blocks=8, apb=8, n=3_000_000, clocks="compressed"),
        # many independent traces at once: 24 traces of 10k-1M events, 64-4096 warps, 16 lanes
        dict(name="batch_24", kind="batch", traces=24, n_min=10_000, n_max=1_000_000, lanes=16),
        # the ranker in use: location features and scores of a trace, then the ranked analysis
        dict(name="ranked_64warp_1M", kind="ranked", blocks=8, apb=8, n=1_000_000),
        # the ranker's training: scores, one gradient, and mini-batch Adam epochs over labelled rows
        dict(name="ranker_fit_40k", kind="fit", rows=40_013, batch=1024, epochs=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    r = rng.random()
    if r < 0.10:
        blocks, apb = rng.choice([(8, 8), (1, 24), (4, 16), (5, 7), (16, 8)])
        return dict(kind="noalloc", blocks=blocks, apb=apb, n=_log(rng, 10_000, 180_000))
    if r < 0.24:
        blocks, apb = rng.choice([(1, 64), (1, 32), (2, 96), (3, 50), (1, 256), (4, 128), (1, 1024)])
        return dict(kind="trace", mix="thread", blocks=blocks, apb=apb, n=_log(rng, 10_000, 600_000))
    if r < 0.32:
        return dict(kind="batch", traces=rng.randint(4, 32), n_min=10_000, n_max=_log(rng, 50_000, 1_500_000),
                    lanes=rng.choice([1, 8, 16]))
    if r < 0.40:
        return dict(kind="ranked", blocks=8, apb=rng.choice([8, 4, 13]), n=_log(rng, 50_000, 2_000_000))
    if r < 0.46:
        return dict(kind="fit", rows=_log(rng, 2_000, 200_000), batch=rng.choice([256, 1000, 4096]), epochs=2)
    if r < 0.54:
        return dict(kind="trace", mix="8192", blocks=rng.choice([256, 200, 129]), apb=32, n=_log(rng, 1_000_000, 40_000_000))
    if r < 0.64:
        blocks, apb = rng.choice([(8, 8), (16, 8), (12, 9), (32, 8)])
        c = dict(kind="trace", mix="64", blocks=blocks, apb=apb, n=_log(rng, 10_000, 5_000_000))
        c.update(rng.choice([dict(clocks="compressed"), dict(hb_only=True), dict(forced=True), dict(check="chunked")]))
        return c
    blocks, apb = rng.choice([(8, 8), (16, 8), (32, 8), (64, 8), (64, 16), (64, 32), (128, 32), (6, 16), (11, 5),
                              (40, 24), (100, 20)])
    c = dict(kind="trace", mix="64", blocks=blocks, apb=apb,
             n=_log(rng, 10_000, 10_000_000) if blocks * apb <= 512 else _log(rng, 100_000, 4_000_000))
    if rng.random() < 0.3:
        c["host"] = True
    return c


def _params(case):
    mix = {"64": MIX64, "8192": MIX8192, "thread": MIXTHREAD}[case.get("mix", "64")]
    p = dict(mix)
    p.update(n_events=case["n"], num_blocks=case["blocks"], agents_per_block=case["apb"])
    if mix is MIX64:  # as the batched workload: a tenth as many address ranks as events
        p["n_ranks"] = max(1000, case["n"] // 10)
    elif mix is MIX8192:
        p["n_ranks"] = max(200_000, int(case["n"] * 0.32))
    elif case["n"] > 20_000 or case["blocks"] > 1:  # more addresses and locks than the 10k-event trace has
        p.update(n_ranks=max(16, case["n"] // 20), zipf_s=1.05, n_locks=32, p_barrier=0.001)
    return p


def _trace(case, seed):
    ev, geo, _ = tracegen.generate(seed, **_params(case))
    return ev, geo.astuple()


def _room(case):
    """Races a caller makes room for."""
    return 3 * case["n"] + 1024 if case.get("mix", "64") != "8192" else 200_000


def _on_gpu(ev):
    return torch.from_numpy(ev.view(np.uint8)).cuda()


def _table(rows):
    """A caller's result array, kept from call to call: (earlier, later) per race, zeros behind them."""
    return np.zeros((rows, 2), dtype=np.int64)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fit":
        rng = np.random.default_rng(seed)
        x = np.abs(rng.normal(0, 1.5, (case["rows"], gwcp.RANK_FEATURES))).astype(np.float32)
        y = ((x[:, 2] * x[:, 14] + 0.3 * rng.normal(size=case["rows"])) > 2.5).astype(np.float32)
        theta = ranker.init_theta(seed)
        return dict(case=case, theta=torch.from_numpy(theta).cuda(), x=torch.from_numpy(x).cuda(),
                    y=torch.from_numpy(y).cuda())
    if kind == "batch":
        # lengths and widths are the case's, the events the seed's
        specs = tracegen.many_specs(case["traces"], case["traces"], case["n_min"], case["n_max"])
        for i, spec in enumerate(specs):
            spec["seed"] = seed * 100_003 + i
        traces = tracegen.generate_many(specs)
        caps = [3 * len(ev) + 1024 for ev, _ in traces]
        outs = [_table(c) for c in caps]
        return dict(case=case, pool=gwcp.Pool(0, lanes=case["lanes"]), caps=caps, outs=outs,
                    traces=[(_on_gpu(ev), geo.astuple()) for ev, geo in traces])
    ev, geo = _trace(case, seed)
    if kind == "noalloc":
        cap = 3 * case["n"] + 1024
        gwcp.analyze_noalloc(0, 0, *geo, 0, 0)  # reserves the scratch, as a caller does at start-up
        return dict(case=case, ev=_on_gpu(ev), geo=geo, n=len(ev), cap=cap,
                    races=torch.zeros((cap, 2), dtype=torch.int64, device="cuda"))
    if kind == "ranked":
        theta = ranker.load_weights()
        if theta is None:
            theta = ranker.init_theta(7)
        plain, ranked = gwcp.Context(0), gwcp.Context(0)
        ranked.set_ranker(theta)
        return dict(case=case, ev=_on_gpu(ev), geo=geo, plain=plain, ranked=ranked, theta=torch.from_numpy(theta).cuda(),
                    out=_table(_room(case)), features=torch.zeros((case["n"], gwcp.RANK_FEATURES), device="cuda"),
                    keys=torch.zeros(case["n"], dtype=torch.int64, device="cuda"),
                    scores=torch.zeros(case["n"], device="cuda"))
    ctx = gwcp.Context(0, hb_only=bool(case.get("hb_only")), forced_barrier=bool(case.get("forced")))
    if case.get("clocks") == "compressed":
        ctx.set_clock_mode(gwcp.CLOCKS_COMPRESSED)
    if case.get("check") == "chunked":
        ctx.set_check_mode(gwcp.CHECK_CHUNKED)
    out = _table(_room(case))
    if case.get("host"):
        pinned = torch.from_numpy(ev.view(np.uint8)).pin_memory()
        return dict(case=case, ctx=ctx, ev=pinned.numpy().view(tracegen.EVENT_DTYPE), pinned=pinned, geo=geo, out=out)
    return dict(case=case, ctx=ctx, ev=_on_gpu(ev), geo=geo, out=out)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "trace":
        ctx = state["ctx"]
        ctx.load_trace(state["ev"], *state["geo"])
        ctx.compute_order()
        races = ctx.report_races(out=state["out"].view(np.uint64))
        return dict(races=state["out"], count=len(races))
    if kind == "noalloc":
        rc, total, bad = gwcp.analyze_noalloc(state["ev"].data_ptr(), state["n"], *state["geo"],
                                              state["races"].data_ptr(), state["cap"])
        return dict(rc=rc, bad=ctypes.c_int64(bad).value, races=state["races"], count=total)
    if kind == "batch":
        got = state["pool"].run_batch(state["traces"], state["caps"], [o.view(np.uint64) for o in state["outs"]])
        return dict(races=state["outs"], counts=np.array([(rc, count) for _, rc, count in got]))
    if kind == "ranked":
        plain, ranked = state["plain"], state["ranked"]
        plain.load_trace(state["ev"], *state["geo"])
        plain.compute_order()
        feat, keys = plain.location_features()
        scores = gwcp.rank_scores(state["theta"], feat)
        ranked.load_trace(state["ev"], *state["geo"])
        ranked.compute_order()
        races = ranked.report_races(out=state["out"].view(np.uint64))
        # a caller that keeps tables of all locations it has seen, zeros behind this trace's
        for table, rows in (("features", feat), ("keys", keys), ("scores", scores)):
            state[table][: len(rows)] = rows
        return dict(features=state["features"], keys=state["keys"], scores=state["scores"], races=state["out"],
                    count=len(races))
    theta, x, y = state["theta"].clone(), state["x"], state["y"]
    scores = gwcp.rank_scores(theta, x)
    grad, loss = gwcp.rank_grad(theta, x, y, 4.0)
    losses = gwcp.rank_train(theta, x, y, case["epochs"], case["batch"], 1e-3, 4.0)
    return dict(scores=scores, grad=grad, loss=loss, theta=theta, losses=losses)


def work(case):
    kind = case["kind"]
    if kind == "fit":  # the rows are read for the scores, the gradient and every epoch
        forward = 2 * (16 * 64 + 64 * 64 + 64) * case["rows"]
        return dict(bytes=case["rows"] * 72, flops=forward * (1 + 3 * (1 + case["epochs"])))
    if kind == "batch":
        n = case["traces"] * (case["n_max"] - case["n_min"]) / math.log(case["n_max"] / case["n_min"])
        return dict(bytes=n * (16 + 16 * RACES_WIDE), flops=0)
    n = case["n"]
    per = {"8192": RACES_8192, "thread": RACES_THREAD}.get(case.get("mix"), RACES_64 if case["blocks"] * case["apb"] <= 64 else RACES_WIDE)
    if kind == "ranked":  # the trace, the races, and a feature row, key and score for about n / 5 locations
        return dict(bytes=n * (16 + 16 * per) + n / 5 * 76, flops=n / 5 * 2 * (16 * 64 + 64 * 64 + 64))
    return dict(bytes=n * (16 + 16 * per), flops=0)


# ---- the ranker's numbers in 64 bits --------------------------------------------------
# (race sets are whole numbers and have no such value)


def _bf16(x):
    return torch.from_numpy(np.asarray(x, dtype=np.float64)).to(torch.float32).to(torch.bfloat16).to(torch.float64).numpy()


def _features(ev, apb):
    """Ascending location keys and their 16 features (float64)."""
    op, agent = ev["op"].astype(np.int64), ev["agent"].astype(np.int64)
    step = (op == tracegen.ACQ).astype(np.int64) - (op == tracegen.REL)
    by = np.argsort(agent, kind="stable")
    run_sum = np.cumsum(step[by])
    first = np.r_[True, agent[by][1:] != agent[by][:-1]]
    start = np.maximum.accumulate(np.where(first, np.arange(len(by)), 0))
    depth = np.empty(len(by), dtype=np.int64)
    depth[by] = run_sum - (run_sum[start] - step[by][start])
    acc = np.nonzero(op <= tracegen.ATOMIC)[0]
    shared = ev["space"][acc] == tracegen.SHARED
    blk = agent[acc] // apb
    keys = np.where(shared, np.uint64(1 << 63) | (blk.astype(np.uint64) << np.uint64(40)) | ev["addr"][acc], ev["addr"][acc])
    o = np.argsort(keys, kind="stable")
    acc, keys, blk = acc[o], keys[o], blk[o]
    new = np.r_[True, keys[1:] != keys[:-1]]
    lo = np.nonzero(new)[0]
    g = np.cumsum(new) - 1
    count = lambda m: np.add.reduceat(m.astype(np.float64), lo)  # noqa: E731
    distinct = lambda v: np.bincount(np.unique(g * 64 + v % 64) // 64, minlength=len(lo)).astype(np.float64)  # noqa: E731
    aop, ag = op[acc], agent[acc]
    n, hi = count(np.ones(len(acc))), np.r_[lo[1:], len(acc)] - 1
    atomic, dev = aop == tracegen.ATOMIC, ev["scope"][acc] == tracegen.DEVICE
    wr, ins = aop != tracegen.READ, depth[acc] > 0
    switch = np.r_[False, (ag[1:] != ag[:-1]) & ~new[1:]]
    cswitch = switch & (wr | np.r_[False, wr[:-1]])
    sync = np.nonzero((op == tracegen.ACQ) | (op == tracegen.REL) | (op == tracegen.BARRIER))[0]
    f, last = acc[lo], acc[hi]
    between = np.searchsorted(sync, last, side="right") - np.searchsorted(sync, f, side="left")
    pairs = np.maximum(n - 1, 1)
    F = [np.log1p(n), np.log1p(count(aop == tracegen.READ)), np.log1p(count(aop == tracegen.WRITE)), np.log1p(count(atomic)),
         np.log1p(distinct(ag)), np.log1p(distinct(blk)), count(atomic & ~dev) / n, count(atomic & dev) / n,
         count(ins) / n, (keys[lo] >> np.uint64(63)).astype(np.float64), between / (last - f + 1.0), np.log1p((last - f).astype(np.float64)),
         count(ag == ag[lo][g]) / n, count(switch) / pairs, count(cswitch) / pairs, count(ins & wr) / np.maximum(count(wr), 1)]
    return keys[lo], np.stack(F, axis=1)


def _split(t):
    cut = np.cumsum([64 * 16, 64, 64 * 64, 64, 64])
    w1, b1, w2, b2, w3, b3 = np.split(np.asarray(t, dtype=np.float64), cut)
    return w1.reshape(64, 16), b1, w2.reshape(64, 64), b2, w3, b3[0]


def _forward(t, x):
    w1, b1, w2, b2, w3, b3 = _split(t)
    xb = _bf16(x)
    z1 = xb @ _bf16(w1).T + b1
    h1 = _bf16(np.maximum(z1, 0))
    z2 = h1 @ _bf16(w2).T + b2
    return np.maximum(z2, 0) @ w3 + b3, xb, z1, h1, z2


def _loss_grad(t, x, y, pos):
    _, _, w2, _, w3, _ = _split(t)
    s, xb, z1, h1, z2 = _forward(t, x)
    wt = np.where(y > 0, pos, 1.0)
    ds = wt * (1 / (1 + np.exp(-s)) - y) / len(s)
    dz2 = np.outer(ds, w3) * (z2 > 0)
    dz1 = (dz2 @ _bf16(w2)) * (z1 > 0)
    g = np.concatenate([(dz1.T @ xb).ravel(), dz1.sum(0), (dz2.T @ h1).ravel(), dz2.sum(0), np.maximum(z2, 0).T @ ds, [ds.sum()]])
    return float(np.mean(wt * (np.logaddexp(0, s) - y * s))), g


def exact(case, seed):
    if case["kind"] == "fit":
        rng = np.random.default_rng(seed)
        x = np.abs(rng.normal(0, 1.5, (case["rows"], gwcp.RANK_FEATURES))).astype(np.float32)
        y = ((x[:, 2] * x[:, 14] + 0.3 * rng.normal(size=case["rows"])) > 2.5).astype(np.float64)
        t = ranker.init_theta(seed).astype(np.float64)
        x = x.astype(np.float64)
        loss, grad = _loss_grad(t, x, y, 4.0)
        scores = _forward(t, x)[0]
        m, v, k, losses = np.zeros_like(t), np.zeros_like(t), 0, []
        batches = -(-len(x) // case["batch"])
        for _ in range(case["epochs"]):
            total = 0.0
            for q in range(batches):
                part = slice(q * case["batch"], (q + 1) * case["batch"])
                one, g = _loss_grad(t, x[part], y[part], 4.0)
                g, total, k = g / batches, total + one / batches, k + 1
                m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
                t = t - 1e-3 * (m / (1 - 0.9 ** k)) / (np.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
            losses.append(total)
        return dict(scores=scores, grad=grad, loss=loss, theta=t, losses=np.array(losses))
    if case["kind"] == "ranked":
        ev, geo = _trace(case, seed)
        keys, feat = _features(ev, geo[1])
        theta = ranker.load_weights()
        if theta is None:
            theta = ranker.init_theta(7)
        scores = np.zeros(case["n"])
        scores[: len(keys)] = _forward(theta, feat)[0]
        table = np.zeros((case["n"], gwcp.RANK_FEATURES))
        table[: len(keys)] = feat
        return dict(features=table, keys=None, scores=scores, races=None, count=None)
    return None
