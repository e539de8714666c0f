"""The calls whose speed counts, and their sizes.

A user of this framework runs a request router: every few milliseconds a
batch of prompts arrives, is routed (`route`), perhaps rebalanced, and
committed to the cache indices (`commit`).  Most cases are one such step of a
scheduler that has been running for a while: the caches hold what earlier
batches left, the queues hold work, and the state moves on with every pass.
The rest are the calls that stand alone: hashing prompts into block keys, a
change of the instance set, and the d-choices sweep.

A step case keeps a cycle of batches whose distinct blocks are several times
what the caches hold, so that a pass finds the hits a live trace would show
(shared prefixes, earlier turns of a conversation), inserts the rest and
evicts as much.  The time between batches is taken from the work that the
busiest instance gets, so that its queue is about 80 % busy and never grows
without bound.

Everything the path computes is an integer, so every output is compared
exactly.  `exact` gives the outputs that follow from a closed definition (block
keys and ring positions, the d-choices sweep); a routing step's follow from the
scheduler's whole history, which the test oracle covers.
"""

import ctypes
import math

import numpy as np
import torch

from paper_2602_06502_gb300 import dualmap as D
from paper_2602_06502_gb300.scheduler import Scheduler

MASK64 = (1 << 64) - 1
PHI = 0x9E3779B97F4A7C15

# dm_choice_rule names that a case may state
RULES = {name: i for i, name in enumerate(D.RULE_NAMES)}

STEP = dict(
    kind="step", host=False, instances=8, vnodes=64, block_tokens=16, route_blocks=16, capacity=16384,
    slo_us=2_000_000, rule="dualmap", candidates=2, adapt_step=0, adapt_max=0, rebalance=False, rebalance_flags=0,
    batch=256, batches=32, vocab=32000, touch=0, slots_log2=0, pool=0,
    prompts="prefix", len_lo=128, len_hi=2048, n_prefix=50, zipf=1.0, prefix_lo=256, prefix_hi=1024,
)


def _step(name, **kw):
    return dict(STEP, name=name, **kw)


def listed():
    return [
        # A small router called once per scheduling tick with prompts in host
        # memory, waiting for the decisions: latency and launches.
        _step("host_small", host=True, batch=16, batches=64, capacity=4096),
        # The tiny workload: 8 instances, 256 prompts of 128-2,048 tokens.
        _step("tiny", batch=256, batches=64, capacity=16384),
        # Multi-turn chat: 32 instances, 1,024 prompts per batch, each the
        # whole history plus 50-500 new tokens, up to 20 turns; an SLO tight
        # enough that the less loaded candidate is taken now and then.
        _step("multiturn", instances=32, vnodes=256, slo_us=5_000, batch=1024, batches=32, vocab=128_000,
              capacity=8192, prompts="turns", len_lo=50, len_hi=500, prefix_lo=50, prefix_hi=500, n_prefix=20),
        # Agent / tool calls: 64 instances, 4,096 prompts per batch of 200
        # templates (2k-8k tokens, Zipf 1.2) and 100-1,000 own tokens.
        _step("agent", instances=64, vnodes=256, slo_us=1_000_000, batch=4096, batches=32, capacity=16384,
              prompts="template", len_lo=100, len_hi=1000, n_prefix=200, zipf=1.2, prefix_lo=2048, prefix_hi=8192,
              touch=1 << 20),
        # Long contexts: 128 instances, 512 prompts of 32k-131k tokens (168 MB
        # of tokens a batch), 64 shared 16k prefixes.
        _step("longctx", instances=128, vnodes=256, batch=512, batches=32, capacity=1 << 18, len_lo=32_768,
              len_hi=131_072, n_prefix=64, zipf=0.8, prefix_lo=16_384, prefix_hi=16_384, touch=1 << 20,
              slots_log2=24, pool=16),
        # Follow-up questions on long documents: prompts of 16k-114k tokens of
        # which all but the last turn is cached.
        _step("followup", instances=32, vnodes=256, batch=64, batches=32, capacity=32768, vocab=128_000,
              prompts="turns", len_lo=256, len_hi=2048, prefix_lo=16_384, prefix_hi=98_304, n_prefix=8),
        # A large cluster with hot prefixes, rebalanced after every batch
        # (a few requests migrate in each).
        _step("scaling", instances=256, vnodes=1024, slo_us=1_000_000, batch=4096, batches=24, capacity=4096,
              len_lo=512, len_hi=8192, n_prefix=1000, zipf=1.0, prefix_lo=256, prefix_hi=2048, rebalance=True,
              touch=1 << 20),
        # The same agent traffic under the rule DualMap is compared with:
        # minimum TTFT over every instance, probing all their indices.
        _step("agent_min_ttft", instances=64, vnodes=256, slo_us=1_000_000, rule="min_ttft", batch=4096, batches=32,
              capacity=16384, prompts="template", len_lo=100, len_hi=1000, n_prefix=200, zipf=1.2, prefix_lo=2048,
              prefix_hi=8192, touch=1 << 20),
        # Four candidates instead of two (App. A.8).
        _step("agent_d4", instances=64, vnodes=256, slo_us=1_000_000, candidates=4, batch=4096, batches=32,
              capacity=16384, prompts="template", len_lo=100, len_hi=1000, n_prefix=200, zipf=1.2, prefix_lo=2048,
              prefix_hi=8192, touch=1 << 20),
        # Block keys of a batch of long prompts, as a KV store asks for them.
        dict(kind="hash", name="hash_long", block_tokens=16, route_blocks=16, n=512, len_lo=32_768, len_hi=131_072),
        # An instance leaves, another joins, and a batch of positions is looked
        # up on the new rings.
        dict(kind="ring", name="ring_change", instances=256, vnodes=1024, n=4096),
        # The sweep behind the choice of two candidates: 10,000 trials.
        dict(kind="potc", name="potc", bins=32, per_bin=1000, d=2, trials=10_000),
    ]


# ---------------------------------------------------------------------------
# Drawn cases.

def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _instance_bytes(capacity, touch):
    entries = 1
    while entries < 2 * (capacity + touch):
        entries *= 2
    return max(entries, 1024) * (2 * 16 + 42)


def draw(rng):
    kind = rng.choice(["step"] * 11 + ["host"] * 2 + ["hash"] * 3 + ["ring"] * 2 + ["potc"] * 2)
    if kind == "hash":
        n = _log_int(rng, 1, 4096)
        hi = _log_int(rng, 64, min(131_072, 40_000_000 // n))
        return dict(kind="hash", block_tokens=rng.choice([4, 8, 16, 16, 32, 64]),
                    route_blocks=rng.choice([1, 16, 16, 100, 256]), n=n, len_lo=max(64, hi // rng.randint(1, 16)),
                    len_hi=hi)
    if kind == "ring":
        return dict(kind="ring", instances=_log_int(rng, 3, 256), vnodes=_log_int(rng, 16, 1024),
                    n=_log_int(rng, 1, 65_536))
    if kind == "potc":
        return dict(kind="potc", bins=_log_int(rng, 2, 64), per_bin=_log_int(rng, 10, 1000), d=rng.randint(1, 4),
                    trials=_log_int(rng, 100, 10_000))
    c = dict(STEP, host=kind == "host")
    c["instances"] = _log_int(rng, 8, 256)
    c["vnodes"] = rng.choice([64, 128, 256, 1024])
    c["block_tokens"] = rng.choice([4, 8, 16, 16, 16, 32, 64])
    c["route_blocks"] = rng.choice([4, 16, 16, 64])
    c["slo_us"] = rng.choice([5_000, 50_000, 1_000_000, 2_000_000])
    c["prompts"] = rng.choice(["prefix", "prefix", "template", "turns"])
    tokens = 2_000_000 if c["host"] else 40_000_000   # a batch's tokens at most
    option = "plain" if c["host"] else rng.choice(["plain"] * 5 + ["rebalance", "adaptive", "pair", "cluster", "d"])
    if option in ("cluster", "d"):
        tokens = 8_000_000
    c["batch"] = _log_int(rng, 1, 512 if c["host"] else 4096)
    if c["prompts"] == "prefix":
        hi = _log_int(rng, 256, min(131_072, max(256, tokens // c["batch"])))
        lo = max(64, hi // rng.randint(2, 16))
        c.update(len_lo=lo, len_hi=hi, prefix_lo=max(16, lo // 4), prefix_hi=max(16, hi // rng.randint(2, 8)),
                 n_prefix=_log_int(rng, 1, 1000), zipf=rng.choice([0.0, 0.8, 1.0, 1.2, 1.4]))
        longest = hi
    elif c["prompts"] == "template":
        hi = _log_int(rng, 256, min(65_536, max(256, tokens // c["batch"])))
        own = max(64, hi // rng.randint(2, 16))
        c.update(len_lo=max(32, own // 10), len_hi=own, prefix_lo=max(16, hi // 4), prefix_hi=hi,
                 n_prefix=_log_int(rng, 1, 400), zipf=rng.choice([0.0, 0.8, 1.0, 1.2]))
        longest = hi + own
    else:
        turns = rng.randint(2, 20)
        hi = _log_int(rng, 256, min(98_304, max(256, tokens // c["batch"])))
        own = max(64, hi // rng.randint(2, 2 * turns))
        c.update(len_lo=max(32, own // 10), len_hi=own, prefix_lo=max(64, hi // 8), prefix_hi=hi, n_prefix=turns)
        longest = hi + (turns - 1) * own
    c["batch"] = max(1, min(c["batch"], tokens // longest))
    c["batches"] = max(4, min(32, 800_000_000 // (c["batch"] * longest)))
    if option == "rebalance":
        c.update(rebalance=True, rebalance_flags=rng.choice([0, 0, 1, 2, 3]))
    elif option == "adaptive":
        c.update(adapt_step=rng.choice([16, 32, 64]), adapt_max=rng.choice([256, 1024, 2048]))
    elif option == "pair":
        c["rule"] = rng.choice(["pair_cache_affinity", "pair_least_loaded", "pair_min_ttft", "pair_preble",
                                "cache_affinity"])
    elif option == "cluster":
        c["rule"] = rng.choice(["least_loaded", "min_ttft", "preble"])
        c["batch"] = max(1, min(c["batch"], 4096 * 64 // c["instances"]))
    elif option == "d":
        c["candidates"] = rng.choice([1, 3, 4, 5, 8])
        c["batch"] = max(1, min(c["batch"], 4096 * 4 // c["candidates"]))
    # caches that hold a part of the cycle's distinct blocks
    distinct = 0.6 * c["batch"] * longest * c["batches"] / c["block_tokens"] / c["instances"]
    c["capacity"] = max(256, min(1 << 18, int(distinct * rng.choice([0.05, 0.2, 0.5]))))
    touch = c["batch"] * (longest + 4) // c["block_tokens"] + 1
    while c["instances"] > 8 and c["instances"] * _instance_bytes(c["capacity"], touch) > 24e9:
        c["instances"] //= 2
    return c


# ---------------------------------------------------------------------------
# Prompts: lengths and shared parts on the host, token ids on the device.

def _zipf(n, s, rng, size):
    w = np.arange(1, n + 1, dtype=np.float64) ** -s
    cdf = np.cumsum(w) / w.sum()
    return np.minimum(np.searchsorted(cdf, rng.random(size), side="right"), n - 1)


def _plan(c, seed):
    """Per batch (lengths, shared tokens, where they start in the pool), and the pool's size."""
    rng = np.random.default_rng(seed)
    nb, n = c["batches"], c["batch"]
    if c["prompts"] == "turns":
        # `n` conversations at a time, each taking consecutive batches with a
        # turn per batch (geometric, n_prefix turns at most); a prompt is the
        # conversation's token stream up to its turn
        L = np.zeros((nb, n), np.int64)
        start = np.zeros((nb, n), np.int64)
        p = 0.2 if c["n_prefix"] > 8 else 0.3
        left = np.zeros(n, np.int64)
        base = np.zeros(n, np.int64)
        length = np.zeros(n, np.int64)
        longest = c["prefix_hi"] + (c["n_prefix"] - 1) * c["len_hi"]
        used = 0
        for b in range(nb):
            new = left == 0
            k = int(new.sum())
            turns = np.minimum(rng.geometric(p, n), c["n_prefix"])
            first = rng.integers(c["prefix_lo"], c["prefix_hi"], n, endpoint=True)
            chunk = rng.integers(c["len_lo"], c["len_hi"], n, endpoint=True)
            if b == 0:   # conversations already under way
                turns = np.maximum(1, turns - rng.integers(0, c["n_prefix"], n) // 2)
            base[new] = used + np.arange(k) * longest
            used += k * longest
            length = np.where(new, first, length + chunk)
            left = np.where(new, turns, left) - 1
            L[b], start[b] = length, base
        # streams packed to the length they reach
        starts, inv = np.unique(start, return_inverse=True)
        reach = np.zeros(len(starts), np.int64)
        np.maximum.at(reach, inv.reshape(-1), L.reshape(-1))
        packed = np.cumsum(reach) - reach
        start = packed[inv.reshape(start.shape)]
        return [(L[b], L[b], start[b]) for b in range(nb)], int(reach.sum())
    plen = rng.integers(c["prefix_lo"], c["prefix_hi"], c["n_prefix"], endpoint=True)
    pstart = np.cumsum(plen) - plen
    out = []
    for _ in range(nb):
        p = _zipf(c["n_prefix"], c["zipf"], rng, n)
        own = rng.integers(c["len_lo"], c["len_hi"], n, endpoint=True)
        L = plen[p] + own if c["prompts"] == "template" else own
        L = np.maximum(L, c["block_tokens"])
        out.append((L, np.minimum(plen[p], L), pstart[p]))
    return out, int(plen.sum())


def _layout(L):
    """16-byte-aligned prompt offsets and the buffer's extent."""
    room = (L + 3) // 4 * 4
    return np.cumsum(room) - room, int(room.sum())


def _fill(L, shared, start, pool, vocab, gen):
    """One batch's token buffer on the device: shared parts from the pool, the rest drawn."""
    off, total = _layout(L)
    dev = pool.device
    tok = torch.randint(vocab, (total,), dtype=torch.int32, device=dev, generator=gen)
    if len(pool) and shared.any():
        room = torch.from_numpy(np.diff(np.append(off, total))).to(dev)
        toff, tsh, tst = (torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (off, shared, start))
        r = torch.repeat_interleave(torch.arange(len(L), device=dev), room, output_size=total)
        pos = torch.arange(total, device=dev) - toff[r]
        tok = torch.where(pos < tsh[r], pool[(tst[r] + pos).clamp_(max=len(pool) - 1)], tok)
    return tok, off, total


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _check(rc, what):
    if rc:
        raise D.DualMapError(rc, what)


# ---------------------------------------------------------------------------
# Scheduler steps.

OUTS = [("cand1", torch.int32), ("cand2", torch.int32), ("hit1", torch.int32), ("hit2", torch.int32),
        ("ttft1", torch.int64), ("ttft2", torch.int64), ("chosen", torch.int32), ("switched", torch.uint8)]


def _prepare_step(c, seed):
    plan, pool_n = _plan(c, seed)
    gen = _gen(seed)
    pool = torch.randint(c["vocab"], (pool_n,), dtype=torch.int32, device="cuda", generator=gen)
    batches = []
    for L, shared, start in plan:
        tok, off, total = _fill(L, shared, start, pool, c["vocab"], gen)
        t_off, t_len = torch.from_numpy(off), torch.from_numpy(L.astype(np.int32))
        if c["host"]:
            batches.append((tok.cpu().pin_memory(), t_off.pin_memory(), t_len.pin_memory(), total))
        else:
            batches.append((tok, t_off.cuda(), t_len.cuda(), total))
    del pool
    s = Scheduler(block_tokens=c["block_tokens"], route_prefix_blocks=c["route_blocks"], vnodes=c["vnodes"],
                  max_instances=c["instances"], capacity=c["capacity"], slo_us=c["slo_us"], max_batch=c["batch"],
                  max_batch_tokens=max(max(b[3] for b in batches), c["block_tokens"]),
                  max_touch_per_instance=c["touch"], index_slots_log2=c["slots_log2"], rebuild_pool=c["pool"],
                  choice_rule=RULES[c["rule"]], candidates=c["candidates"], adapt_step_blocks=c["adapt_step"],
                  adapt_max_blocks=c["adapt_max"], adapt_window=4 if c["adapt_step"] else 1,
                  rebalance_flags=c["rebalance_flags"], seed=seed)
    for i in range(c["instances"]):
        _check(s.add_instance(i), "dm_add_instance")
    state = {"s": s, "batches": batches, "n": c["batch"], "k": 0, "t": 0, "gap": 0, "rebalance": c["rebalance"],
             "d": c["candidates"] != 2, "host": c["host"]}
    if c["host"]:
        state["out"] = {k: torch.zeros(c["batch"], dtype=t).pin_memory() for k, t in OUTS}
        state["out_struct"] = D.make_out(*[state["out"][k] for k, _ in OUTS])
    # the cycle once with every queue run empty between batches: the caches
    # fill, and the work each instance gets per batch gives the batch interval
    work = np.zeros(c["instances"], np.float64)
    state["gap"] = 1 << 40
    for _ in batches:
        _pass(state)
        work += s.loads()[:c["instances"]].astype(np.float64)
    state["gap"] = int(1.25 * work.max() / len(batches)) + 1
    for _ in batches:   # once more at that pace: queues as they stand in service
        _pass(state)
    _check(s.last_error(), "preparing the scheduler")
    return state


def _pass(st):
    s, n = st["s"], st["n"]
    tok, off, lens, total = st["batches"][st["k"]]
    st["k"] = (st["k"] + 1) % len(st["batches"])
    st["t"] += st["gap"]
    if st["host"]:
        b = D.make_batch(tok, off, lens, n, total, st["t"])
        _check(D.dm_route_batch_host(s.h, b, st["out_struct"]), "dm_route_batch_host")
        s.commit()
        return st["out"]
    if st["d"]:
        s.route_d(tok, off, lens, n, total, st["t"])
        s.commit()
        return s.out_d
    s.route(tok, off, lens, n, total, st["t"])
    if st["rebalance"]:
        s.rebalance()
        s.commit()
        return {**s.out, "migrations": s.mig, "migrations_n": s.mig_n}
    s.commit()
    return s.out


# ---------------------------------------------------------------------------
# Stand-alone calls.

def _hash_inputs(c, seed):
    rng = np.random.default_rng(seed)
    L = np.maximum(rng.integers(c["len_lo"], c["len_hi"], c["n"], endpoint=True), c["block_tokens"])
    off, total = _layout(L)
    tok = torch.randint(128_000, (total,), dtype=torch.int32, device="cuda", generator=_gen(seed))
    return L, off, total, tok


def _key_room(c):
    """Entries of the key buffer: enough for prompts of these lengths, whatever they are."""
    return c["n"] * max(1, c["len_hi"] // c["block_tokens"])


def _prepare_hash(c, seed):
    L, off, total, tok = _hash_inputs(c, seed)
    s = Scheduler(block_tokens=c["block_tokens"], route_prefix_blocks=c["route_blocks"], max_instances=2,
                  capacity=1024, max_batch=c["n"], max_batch_tokens=total, max_touch_per_instance=1024, seed=seed)
    return {"s": s, "n": c["n"], "total": total, "tok": tok, "off": torch.from_numpy(off).cuda(),
            "len": torch.from_numpy(L.astype(np.int32)).cuda(),
            "keys": torch.zeros(_key_room(c), dtype=torch.int64, device="cuda"),
            "key_off": torch.zeros(c["n"] + 1, dtype=torch.int64, device="cuda"),
            "pos": torch.zeros(2 * c["n"], dtype=torch.int64, device="cuda")}


def _run_hash(st):
    b = D.make_batch(st["tok"], st["off"], st["len"], st["n"], st["total"], 0)
    _check(D.dm_hash_prompts(st["s"].h, b, st["keys"], st["key_off"], st["pos"]), "dm_hash_prompts")
    return {"keys": st["keys"], "key_off": st["key_off"], "pos": st["pos"]}


def _prepare_ring(c, seed):
    s = Scheduler(vnodes=c["vnodes"], max_instances=c["instances"] + 1, capacity=16384, max_batch=1024,
                  max_batch_tokens=1 << 20, max_touch_per_instance=16384, seed=seed)
    for i in range(c["instances"] + 1):
        _check(s.add_instance(i), "dm_add_instance")
    rng = np.random.default_rng(seed)
    out = int(rng.integers(c["instances"] + 1))
    _check(s.remove_instance(out), "dm_remove_instance")
    pos = torch.from_numpy(rng.integers(-(1 << 63), (1 << 63) - 1, 2 * c["n"], dtype=np.int64)).cuda()
    return {"s": s, "n": c["n"], "m": c["instances"] + 1, "out": out, "pos": pos,
            "o1": torch.zeros(c["n"], dtype=torch.int32, device="cuda"),
            "o2": torch.zeros(c["n"], dtype=torch.int32, device="cuda")}


def _run_ring(st):
    s, back = st["s"], st["out"]
    st["out"] = (back + 1) % st["m"]
    _check(s.remove_instance(st["out"]), "dm_remove_instance")
    _check(s.add_instance(back), "dm_add_instance")
    _check(D.dm_ring_lookup(s.h, st["pos"], st["n"], st["o1"], st["o2"]), "dm_ring_lookup")
    return {"owner1": st["o1"], "owner2": st["o2"]}


def _prepare_potc(c, seed):
    return {"c": c, "seed": seed, "out": torch.zeros(c["trials"], dtype=torch.int32, device="cuda")}


def _run_potc(st):
    c = st["c"]
    _check(D.dm_potc_max_loads(c["bins"], c["bins"] * c["per_bin"], c["d"], c["trials"], st["seed"], st["out"],
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "dm_potc_max_loads")
    return st["out"]


# ---------------------------------------------------------------------------
# The interface.

def prepare(case, seed):
    return {"step": _prepare_step, "hash": _prepare_hash, "ring": _prepare_ring, "potc": _prepare_potc}[case["kind"]](
        case, int(seed))


def run(state):
    if "batches" in state:
        return _pass(state)
    if "keys" in state:
        return _run_hash(state)
    if "o1" in state:
        return _run_ring(state)
    return _run_potc(state)


def work(case):
    """Bytes that one pass has to read and write, and its integer operations."""
    c = case
    if c["kind"] == "potc":
        balls = c["bins"] * c["per_bin"] * c["trials"]
        return {"bytes": 4 * c["trials"], "flops": 12 * c["d"] * balls}   # SplitMix64, scaling, compare
    if c["kind"] == "ring":
        # both rings written with the change (12 bytes a node), positions and owners
        return {"bytes": 2 * 2 * 12 * 2 * c["instances"] * c["vnodes"] + 24 * c["n"], "flops": 0}
    if c["kind"] == "hash":
        tokens = c["n"] * (c["len_lo"] + c["len_hi"]) / 2
        return {"bytes": 4 * tokens + 8 * tokens / c["block_tokens"], "flops": 2 * tokens}
    plan, _ = _plan(c, 0)
    tokens = float(np.mean([p[0].sum() for p in plan]))
    # tokens in; per block one index slot read and written and one log record
    # written; per request its layout, outputs and queue entry
    bytes_ = 4 * tokens + tokens / c["block_tokens"] * (16 + 16 + 16) + c["batch"] * (12 + 33 + 64)
    if c["rule"] in ("least_loaded", "min_ttft", "preble"):   # a first-block probe on every instance
        bytes_ += 16 * c["batch"] * c["instances"]
    return {"bytes": bytes_, "flops": 2 * tokens}


def tolerance(case):
    """Everything is integer arithmetic with fixed tie rules."""
    return "exact"


# ---------------------------------------------------------------------------
# Closed definitions, in 64-bit integer arithmetic.

def _mix(x):
    """MurmurHash3's 64-bit finaliser on int64 tensors (arithmetic mod 2^64)."""
    for m in (0xFF51AFD7ED558CCD, 0xC4CEB9FE1A85EC53):
        x = (x ^ ((x >> 33) & 0x7FFFFFFF)) * _signed(m)
    return x ^ ((x >> 33) & 0x7FFFFFFF)


def _signed(u):
    u &= MASK64
    return u - (1 << 64) if u >> 63 else u


def _split_next(state):
    state = (state + PHI) & MASK64
    z = state
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & MASK64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & MASK64
    return state, z ^ (z >> 31)


def _exact_hash(c, seed):
    B = c["block_tokens"]
    L, off, _, tok = _hash_inputs(c, seed)
    words, state = [], seed
    for _ in range(2 * B + 5):
        state, w = _split_next(state)
        words.append(w)
    k1, k2 = (torch.tensor([w & 0xFFFFFFFF for w in words[i * B:(i + 1) * B]], device="cuda") for i in (0, 1))
    g1, g2 = words[2 * B] | 1, words[2 * B + 1] | 1
    sc, sr1, sr2 = (_signed(w) for w in words[2 * B + 2:2 * B + 5])
    nblk = L // B
    key_off = np.concatenate([[0], np.cumsum(nblk)])
    keys = torch.zeros(_key_room(c), dtype=torch.int64, device="cuda")
    pos = torch.zeros(2 * len(L), dtype=torch.int64, device="cuda")

    def digests(t, k, g):   # NH over each block's token pairs, then the block's digest
        x = (t + k) & 0xFFFFFFFF
        nh = (x[:, 0::2] * x[:, 1::2]).sum(1)
        return _mix(nh + torch.arange(1, len(t) + 1, device="cuda") * _signed(g))

    for r in range(len(L)):
        nb = int(nblk[r])
        t = tok[int(off[r]):int(off[r]) + nb * B].to(torch.int64).reshape(nb, B)
        chain = torch.cumsum(digests(t, k1, g1), 0)
        key = _mix(chain ^ sc)
        keys[int(key_off[r]):int(key_off[r + 1])] = torch.where(key == 0, 1, key)
        K = min(c["route_blocks"], nb)
        pos[2 * r] = _mix(chain[K - 1:K] ^ sr1)[0]
        pos[2 * r + 1] = _mix(digests(t[:K], k2, g2).sum().reshape(1) ^ sr2)[0]
    return {"keys": keys, "key_off": torch.from_numpy(key_off).cuda(), "pos": pos}


def _exact_potc(c, seed):
    n, d, T = c["bins"], c["d"], c["trials"]
    m = n * c["per_bin"]
    if m * d > 100_000:
        return None
    load = torch.zeros(T, n, dtype=torch.int64, device="cuda")
    rows = torch.arange(T, device="cuda")
    one = torch.ones(T, 1, dtype=torch.int64, device="cuda")
    ks = torch.arange(d, device="cuda")

    def shift(z, k):   # logical right shift
        return (z >> k) & ((1 << (64 - k)) - 1)

    for t in range(m):
        # the (c+1)-th SplitMix64 output, c = (s m + t) d + k, scaled to a bin
        z = ((rows * m + t) * d)[:, None] + ks + 1
        z = z * _signed(PHI) + _signed(seed)
        z = (z ^ shift(z, 30)) * _signed(0xBF58476D1CE4E5B9)
        z = (z ^ shift(z, 27)) * _signed(0x94D049BB133111EB)
        z = z ^ shift(z, 31)
        bins = shift(shift(z, 32) * n + shift((z & 0xFFFFFFFF) * n, 32), 32)   # floor(z n / 2^64)
        loads = load.gather(1, bins)
        best = bins.gather(1, (loads * d + ks).argmin(1, keepdim=True))   # ties to the earlier choice
        load.scatter_add_(1, best, one)
    return load.max(1).values.to(torch.int32)


def exact(case, seed):
    if case["kind"] == "hash":
        return _exact_hash(case, int(seed))
    if case["kind"] == "potc":
        return _exact_potc(case, int(seed))
    return None
