"""Timed cases: what a program that samples random tilings has the library do.

Each case is one pass through the public Python entry points, over the sizes
of the workloads that bench.py, serve.py and the tests use: chains on Aztec
diamonds, rectangles, lozenge hexagons and the domain-wall square at uniform,
per-site and table thresholds, batches of uneven chains, and the two exact
samplers.  A pass leaves its results on the device, as the benchmark does.

`work` counts the bytes a pass cannot do without (start state and thresholds
read once, results written once; sweeps keep the state on chip) and, under
"flops", its 32-bit integer operations: about 80 per Philox4x32-10 call, one
call per 128 sites and random bit plane, and the bitwise site updates.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

import paper_1804_07250_gb300 as T
from paper_1804_07250_gb300 import serve

_PROGRAM = []


def _program():
    """The program's one context and stream."""
    if not _PROGRAM:
        _PROGRAM.extend([T.Context(0), torch.cuda.Stream()])
    return _PROGRAM


def listed():
    return [
        # A small diamond advanced a little and looked at (the order-32
        # workload, an interactive picture): launches and latency count.
        dict(name="aztec32_uniform", kind="chain", domain="aztec", a=32, b=0, c=0, weights="uniform", order="fixed",
             sweeps=100, stride=0, resume=False),
        # The benchmark's default workload, fewer sweeps: a large uniform
        # diamond with density samples, heights and domino type densities.
        dict(name="aztec2048_uniform_density", kind="chain", domain="aztec", a=2048, b=0, c=0, weights="uniform",
             order="fixed", sweeps=6000, stride=100, resume=False),
        # RandomWalk as printed (a random colour every step) on an N x N
        # square, flips counted: the acceptance rate of a study of mixing.
        dict(name="rect1000_random_order", kind="chain", domain="rect", a=1000, b=999, c=0, weights="uniform",
             order="random", sweeps=1000, stride=0, resume=False),
        # Dominoes with random edge weights (the served and batched kind) on
        # a diamond of a size between the powers of two.
        dict(name="aztec1333_edge_weights", kind="chain", domain="aztec", a=1333, b=0, c=0, weights="site",
             order="fixed", sweeps=300, stride=0, resume=True),
        # The lozenge workload of the benchmark: q^volume on the largest box.
        dict(name="hexagon1024_q", kind="chain", domain="hexagon", a=1024, b=1024, c=1024, weights="q", order="fixed",
             sweeps=1500, stride=0, resume=True),
        # A served lozenge request: independent sides, a weight per vertex.
        dict(name="hexagon_ragged_volume", kind="chain", domain="hexagon", a=301, b=467, c=214, weights="site",
             order="fixed", sweeps=1000, stride=0, resume=True),
        # The six-vertex workload of the benchmark (a = b = 1, c = sqrt 2).
        dict(name="dwbc2048_sqrt2", kind="chain", domain="dwbc", a=2048, b=0, c=0, weights="sqrt2", order="fixed",
             sweeps=1500, stride=0, resume=True),
        # A served six-vertex request: six unequal weights, ordinary size.
        dict(name="dwbc333_table", kind="chain", domain="dwbc", a=333, b=0, c=0, weights="table", order="fixed",
             sweeps=1000, stride=0, resume=True),
        # Many weighted diamonds of uneven size advanced together (the
        # batched workload, fewer chains), autotuned, in graph blocks; every
        # sample is read out.
        dict(name="batch_aztec_edge_weights", kind="batch", chains=128, lo=16, hi=512, sweeps=500),
        # One stretch of the serving loop: a mix of requests, plain launches.
        dict(name="serve_mix", kind="serve", chains=12, hi=1024, sweeps=100),
        # One exact uniform sample of the order-2048 diamond by shuffling.
        dict(name="shuffle2048", kind="shuffle", a=2048),
        # One exact sample by coupling from the past.
        dict(name="cftp_aztec96", kind="cftp", a=96),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    r = rng.random()
    if r < 0.7:
        c = dict(kind="chain", a=0, b=0, c=0, order="fixed", sweeps=_logint(rng, 50, 800), stride=0, resume=False)
        d = c["domain"] = rng.choice(["aztec", "aztec", "aztec", "rect", "hexagon", "hexagon", "dwbc", "dwbc"])
        if d == "aztec":
            c["a"] = _logint(rng, 16, 2048)
            c["weights"] = rng.choice(["uniform", "site"])
            if c["weights"] == "uniform" and rng.random() < 0.5:
                c["stride"] = rng.randint(1, 100)
            c["resume"] = c["weights"] == "site"
        elif d == "rect":
            c["a"], c["b"] = 2 * _logint(rng, 16, 700), _logint(rng, 16, 1400)
            c["weights"] = "uniform"
            c["order"] = rng.choice(["fixed", "random"])
        elif d == "hexagon":
            c["a"], c["b"], c["c"] = (_logint(rng, 16, 800) for _ in range(3))
            c["weights"] = rng.choice(["uniform", "q", "site"])
            c["resume"] = True
        else:
            c["a"] = _logint(rng, 32, 2048)
            c["weights"] = rng.choice(["uniform", "sqrt2", "table"])
            c["resume"] = True
        return c
    if r < 0.8:
        hi = rng.randint(64, 512)
        return dict(kind="batch", chains=rng.randint(16, 96), lo=16, hi=hi, sweeps=rng.randint(50, 450))
    if r < 0.85:
        return dict(kind="serve", chains=rng.randint(4, 10), hi=rng.randint(128, 900), sweeps=rng.randint(40, 99))
    if r < 0.95:
        return dict(kind="shuffle", a=_logint(rng, 32, 1900))
    return dict(kind="cftp", a=rng.randint(16, 64))


# ---------------------------------------------------------------------------
# What a program has in hand before the call.
# ---------------------------------------------------------------------------
_BURN = 3000      # sweeps that take a chain away from its frozen start


def _domain(case):
    d = case["domain"]
    if d == "aztec":
        return T.Domain.aztec(case["a"])
    if d == "rect":
        return T.Domain.rect(case["a"], case["b"])
    if d == "hexagon":
        return T.Domain.hexagon(case["a"], case["b"], case["c"])
    return T.Domain.dwbc(case["a"])


def _thresholds(case, dom, seed, stream):
    w = case["weights"]
    if w == "site":
        t = torch.empty((dom.info.height, dom.info.width), dtype=torch.int32, device="cuda")
        dom.lognormal_thresholds_device(0.5, seed, t, stream=stream)
        stream.synchronize()
        return T.thresholds(site=t)
    if w == "q":
        return T.thresholds(scalar=T.lozenge_thresholds(0.9995)[0])
    if case["domain"] == "dwbc":
        if w == "sqrt2":
            w6 = [1.0, 1.0, 1.0, 1.0, 2.0 ** 0.5, 2.0 ** 0.5]
        elif w == "table":
            w6 = np.exp(0.5 * np.random.default_rng([seed, 6]).standard_normal(6))
        else:
            w6 = np.ones(6)
        return T.thresholds(table16=T.sixv_thresholds(w6))
    return T.thresholds(scalar=1 << 31)


def prepare(case, seed):
    """Inputs and handles of one case.  Only the seed varies them: sizes (and
    a batch's mix of sizes and weights) come from the case."""
    ctx, stream = _program()
    kind = case["kind"]
    if kind == "chain":
        dom = _domain(case)
        chain = T.Chain(ctx, dom, seed=seed, stream_id=seed % 1000, th=_thresholds(case, dom, seed, stream))
        if case["order"] == "random":
            chain.set_order(True)
            chain.count_flips(True)
        s = dict(case=case, stream=stream, chain=chain, init=None,
                 state=torch.empty(dom.canon_shape, dtype=torch.uint8, device="cuda"),
                 height=torch.empty(dom.height_shape, dtype=torch.int32, device="cuda"),
                 hash=torch.zeros(1, dtype=torch.int64, device="cuda"), nsew=None)
        if case["resume"]:
            # a configuration saved by an earlier run
            chain.run(_BURN, stream=stream)
            s["init"] = torch.empty(dom.canon_shape, dtype=torch.uint8, device="cuda")
            chain.read_state(s["init"], stream=stream)
            chain.sync(stream)
        if case["stride"]:
            s["nsew"] = torch.empty((4, dom.info.height - 1, dom.info.width - 1), dtype=torch.float64, device="cuda")
        return s
    if kind == "batch":
        # the orders belong to the case, the weights and the chains' randomness to the seed
        rng = np.random.default_rng([case["chains"], case["lo"], case["hi"]])
        chains = []
        for i, n in enumerate(rng.integers(case["lo"], case["hi"] + 1, size=case["chains"])):
            dom = T.Domain.aztec(int(n))
            th = _thresholds(dict(weights="site"), dom, seed * 1000 + i, stream)
            chains.append(T.Chain(ctx, dom, seed=seed, stream_id=i, th=th))
        batch = T.Batch(ctx, chains)
        batch.autotune(16, stream=stream)
        batch.set_plan(graph_block=100)
        batch.run(300, stream=stream)
        return _batch_state(case, stream, batch, None)
    if kind == "serve":
        hi = case["hi"]
        reqs = serve.make_requests(case["chains"], 200.0, hi, aztec=(32, hi), hexagon=(16, hi // 2), dwbc=(32, hi))
        jobs = [serve.build_job(ctx, dataclasses.replace(r, seed=seed), stream) for r in reqs]
        batch = T.Batch(ctx, [j.chain for j in jobs])
        batch.set_plan(128, 4, -1)           # the serving loop's plan
        batch.run(300, stream=stream)
        return _batch_state(case, stream, batch, jobs)
    if kind == "shuffle":
        n = case["a"]
        return dict(case=case, stream=stream, seed=seed,
                    state=torch.empty((2, 2 * n + 1, 2 * n + 1), dtype=torch.uint8, device="cuda"))
    dom = T.Domain.aztec(case["a"])
    return dict(case=case, stream=stream, seed=seed, dom=dom, th=T.thresholds(scalar=1 << 31),
                state=torch.empty(dom.canon_shape, dtype=torch.uint8, device="cuda"))


def _batch_state(case, stream, batch, keep):
    sizes = [int(c.domain.info.canon_bytes) for c in batch.chains]
    states = torch.empty(sum(sizes), dtype=torch.uint8, device="cuda")
    stream.synchronize()
    return dict(case=case, stream=stream, batch=batch, keep=keep, states=states, parts=list(states.split(sizes)),
                hashes=torch.zeros(len(sizes), dtype=torch.int64, device="cuda"))


# ---------------------------------------------------------------------------
# One pass.
# ---------------------------------------------------------------------------
def run(state):
    s, case, stream = state, state["case"], state["stream"]
    kind = case["kind"]
    if kind == "chain":
        chain = s["chain"]
        if s["init"] is None:
            chain.reset(stream=stream)
        else:
            chain.write_state(s["init"], stream=stream)
            chain.seek(_BURN)
        if case["stride"]:
            chain.density_begin(case["stride"], case["sweeps"] // 2)
        if case["order"] == "random":
            chain.count_flips(True)
        chain.run(case["sweeps"], stream=stream)
        chain.read_state(s["state"], stream=stream)
        chain.read_height(s["height"], stream=stream)
        chain.state_hash(out=s["hash"], stream=stream)
        out = [s["state"], s["height"], s["hash"]]
        if case["stride"]:
            out.append(chain.read_nsew(s["nsew"], stream=stream))
        if case["order"] == "random":
            out.append(chain.flips)
        return out
    if kind in ("batch", "serve"):
        batch = s["batch"]
        batch.run(case["sweeps"], stream=stream)
        for chain, part in zip(batch.chains, s["parts"]):
            chain.read_state(part, stream=stream)
        batch.hashes(s["hashes"], stream=stream)
        return [s["states"], s["hashes"]]
    if kind == "shuffle":
        return [T.aztec_shuffle(_program()[0], case["a"], seed=s["seed"], out=s["state"], stream=stream)]
    _, t_used = T.cftp(_program()[0], s["dom"], seed=s["seed"], th=s["th"], t0=64, out=s["state"], stream=stream)
    return [s["state"], t_used]


# ---------------------------------------------------------------------------
# What a pass cannot do without.
# ---------------------------------------------------------------------------
def _sites_box(case):
    d, a, b, c = case["domain"], case["a"], case["b"], case["c"]
    if d == "aztec":
        return a * a + (a - 1) ** 2, (2 * a + 1) ** 2, 2
    if d == "rect":
        return (a - 1) * (b - 1), (a + 1) * (b + 1), 2
    if d == "hexagon":
        return a * b + b * c + c * a - a - b - c + 1, (a + c + 1) * (b + c + 1), 3
    return (a - 1) ** 2, (a + 2) ** 2, 2


def _ops(sites, planes):
    """Integer operations of one sweep: 80 per Philox call, 20 per word of 32 sites."""
    return sites / 128.0 * 80 * planes + sites / 32.0 * 20


def work(case):
    kind = case["kind"]
    if kind == "chain":
        sites, box, types = _sites_box(case)
        nbytes = types * box + 4 * box                       # state and heights out
        nbytes += types * box if case["resume"] else types * box / 8
        nbytes += 4 * box if case["weights"] == "site" else 0
        nbytes += 32 * box if case["stride"] else 0          # four FP64 densities a face
        planes = 1 if case["weights"] == "uniform" and case["domain"] != "dwbc" else 4
        return {"bytes": nbytes, "flops": case["sweeps"] * _ops(sites, planes)}
    if kind == "batch":
        lo, hi, k = case["lo"], case["hi"], case["chains"]
        n2 = (lo * lo + lo * hi + hi * hi) / 3.0             # mean square of the orders
        return {"bytes": k * n2 * 4 * (2 + 4), "flops": k * case["sweeps"] * _ops(2 * n2, 4)}
    if kind == "serve":
        hi, k = case["hi"], case["chains"]
        n2 = hi * hi / 3.0
        return {"bytes": k * n2 * 3 * (2 + 2), "flops": k * case["sweeps"] * _ops(n2, 3)}
    n = case["a"]
    if kind == "shuffle":
        # every step looks at its K^2 blocks of four edges; a sixth of them draw
        blocks = n * (n + 1) * (2 * n + 1) / 6
        return {"bytes": 2 * (2 * n + 1) ** 2, "flops": blocks * 20 / 32 + blocks / 6 * 80}
    # top and bottom chains over T = 64, 128, ..., about 2 n^2 sweeps
    return {"bytes": 2 * (2 * n + 1) ** 2, "flops": 2 * 4 * n * n * _ops(2 * n * n, 1)}


# ---------------------------------------------------------------------------
# The same densities from plain torch: the chain of a uniform Aztec diamond
# with its own Philox, one byte per edge.  States, heights, hashes and flips
# are whole numbers and have no 64-bit value of their own.
# ---------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, k0, k1):
    m = 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & m) ^ c1 ^ k0, p1 & m, ((p0 >> 32) & m) ^ c3 ^ k1, p0 & m
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return torch.stack([c0, c1, c2, c3], -1)


def exact(case, seed):
    if case["kind"] != "chain" or not case["stride"]:
        return None
    n, sweeps = case["a"], case["sweeps"]
    if not torch.cuda.is_available() and n * n * sweeps > 10_000_000:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    W = 2 * n + 1
    hz = torch.zeros((W + 1, W + 2), dtype=torch.bool, device=dev)   # row y at y, column x at x + 1
    vt = torch.zeros((W + 2, W + 1), dtype=torch.bool, device=dev)   # row y at y + 1, column x at x
    for fy in range(2 * n):                                          # rows of faces, horizontal dominoes
        m = fy + 1 if fy < n else 2 * n - fy
        vt[fy + 1, n - m + 1:n + m:2] = True
    kg = -(-((W + 1) // 2) // 128)
    groups = torch.arange(W * kg, device=dev, dtype=torch.int64)[None]
    bit = torch.arange(32, device=dev, dtype=torch.int64)
    chz = torch.zeros(hz.shape, dtype=torch.int32, device=dev)
    cvt = torch.zeros(vt.shape, dtype=torch.int32, device=dev)
    samples, burn = 0, sweeps // 2
    chunk = max(1, min(32, 4_000_000 // (W * kg)))
    for s0 in range(0, sweeps, chunk):
        k = min(chunk, sweeps - s0)
        slot = torch.arange(2 * k, device=dev, dtype=torch.int64)[:, None]
        words = _philox(groups + 0 * slot, s0 + slot // 2 + 0 * groups, slot % 2 + 0 * groups,
                        0 * groups + 0 * slot + seed % 1000, seed & 0xFFFFFFFF, seed >> 32)
        for i in range(2 * k):
            u = ((words[i][..., None] >> bit) & 1).bool().reshape(W, kg * 128)
            for r in (0, 1):                                         # rows of each parity
                x0 = (i + r) % 2
                nx = (W - x0 + 1) // 2
                e, w = hz[r:W:2, x0 + 1:W + 1:2], hz[r:W:2, x0:W:2]
                nn, ss = vt[r + 1:W + 1:2, x0:W:2], vt[r:W:2, x0:W:2]
                up, down = e & w, nn & ss
                flip = torch.where(~u[r::2, :nx], down & ~e & ~w, up & ~nn & ~ss)
                for v in (e, w, nn, ss):
                    v ^= flip
            if i % 2 == 1:
                s = s0 + i // 2 + 1
                if s >= burn and (s - burn) % case["stride"] == 0:
                    chz += hz
                    cvt += vt
                    samples += 1
    hzc, vtc = chz[:W, 1:W + 1].double(), cvt[1:W + 1, :W].double()
    F = W - 1
    y, x = torch.meshgrid(torch.arange(F, device=dev), torch.arange(F, device=dev), indexing="ij")
    left_here = (x + y) % 2 == n % 2                                 # this face has colour kappa
    right, left, top, bottom = vtc[:F, 1:], vtc[:F, :F], hzc[1:, :F], hzc[:F, :F]
    zero = torch.zeros_like(right)
    north = torch.where(left_here, right, zero) + torch.where(~left_here, left, zero)
    south = torch.where(~left_here, right, zero) + torch.where(left_here, left, zero)
    west = torch.where(~left_here, top, zero) + torch.where(left_here, bottom, zero)
    east = torch.where(left_here, top, zero) + torch.where(~left_here, bottom, zero)
    return [None, None, None, torch.stack([north, south, east, west]) / max(1, samples)]
