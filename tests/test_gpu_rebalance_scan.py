"""Rebalancing with more hotspots than the scan keeps targets for (128) and
more instances than its mask has bits (64): hotspots that could move nothing
under the loads at the call's start, and do so after an earlier hotspot gave
work away, are visited; loads and works below and past 32 bits.  Bit for bit
against the oracle, whose migrations also show that the batch has such
hotspots."""

import numpy as np
import pytest

from parity_harness import Pair, lib_ready
from tracegen import workload

pytestmark = pytest.mark.gpu

N, TOP, MID, B = 560, 40, 220, 16


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


def skewed_batch(ora, seed):
    """Prompts such that 40 instances (top) are the heaviest and can move much
    of their work to idle instances, and 220 (mid) are hot too but have their
    other candidates among the top."""
    rng = np.random.default_rng(seed)
    ids = rng.permutation(N)
    kind = np.zeros(N, int)
    kind[ids[:TOP]], kind[ids[TOP:TOP + MID]] = 2, 1
    starts = rng.integers(0, 32000, (25_000, 2 * B), dtype=np.uint32)   # the routing prefix
    pos = np.array([ora.prompt_keys(x)[1] for x in starts], np.uint64)
    c1, c2 = (ora.ring_owners(pos[:, f].copy(), f) for f in (0, 1))
    prompts = []
    for i in ids[:TOP + MID]:
        own = np.nonzero((c1 == i) & (kind[c2] == (2 if kind[i] == 1 else 0)))[0]
        for _ in range(int(rng.integers(30, 36) if kind[i] == 2 else rng.integers(14, 19)) if len(own) else 0):
            rest = rng.integers(0, 32000, int(rng.integers(8 * B, 12 * B)), dtype=np.uint32)
            prompts.append(np.concatenate([starts[rng.choice(own)], rest]))
    prompts = [prompts[k] for k in rng.permutation(len(prompts))]
    lens = np.array([len(p) for p in prompts], np.uint32)
    room = (lens.astype(np.uint64) + 3) // 4 * 4
    off = np.cumsum(room) - room
    tok = np.zeros(int(room.sum()), np.uint32)
    for p, o in zip(prompts, off):
        tok[int(o):int(o) + len(p)] = p
    return tok, off.astype(np.uint64), lens


def scan(out, lens, W, cost, slo):
    """Hotspots by (load descending, id), their ranks, and those with a request that may move under these loads."""
    W = [int(w) for w in W]
    total = sum(W)
    hot = sorted((i for i in range(N) if 2 * W[i] * N > 3 * total), key=lambda i: (-W[i], i))
    rank = {i: k for k, i in enumerate(hot)}
    ahead, now = [0] * N, set()
    for r in range(len(lens)):
        i = int(out["chosen"][r])
        j = int(out["cand2"][r]) if i == out["cand1"][r] else int(out["cand1"][r])
        own = cost * int(lens[r])
        ahead[i] += own
        if i in rank and ahead[i] > W[j] + own and W[j] + own < slo:
            now.add(i)
    return hot, rank, now


@pytest.mark.parametrize("cost,seed", [(1, 1), (1, 2), (1 << 26, 3)])
def test_hotspots_that_may_move_later(cost, seed):
    slo = 30_000 * cost
    w = workload("tiny", n_instances=N, vnodes=32, slo_us=slo, cost_us=cost, batch=8192, capacity=4096, block_tokens=B,
                 route_prefix_blocks=2)
    p = Pair(w, max_instances=N, max_batch_tokens=1 << 22, max_touch=1 << 15, max_queue=1024, choice_rule=5)
    for i in range(N):
        assert p.add(i) == 0
    tok, off, lens = skewed_batch(p.ora, seed)
    out = p.route(tok, off, lens, 1)
    assert not (out["hit1"].any() or out["hit2"].any())
    before = p.ora.loads()
    hot, rank, now = scan(out, lens, before, cost, slo)
    assert p.rebalance() > 0
    after = p.ora.loads()
    gave = {i for i in hot if after[i] < before[i]}
    woken = [i for i in gave if i not in now]
    assert len(hot) > 128 and any(rank[i] < 128 for i in woken)
    assert any(rank[i] >= 128 for i in woken) and any(i not in gave for i in hot[128:])
    p.commit()
    p.check_state(tag="end")
    p.gpu.close()


@pytest.mark.parametrize("share,slo", [((3000,), 1 << 30), ((3000, 900, 700), 20_000), ((1200, 1000, 900, 0, 40), 1 << 30),
                                       ((2500, 2400), 1)])
def test_hotspots_with_long_queues(share, slo):
    """Hotspots with more than 256 entries for each hotspot (visited without a
    scan) beside ones with fewer, over two batches."""
    n = sum(share)
    w = workload("tiny", n_instances=8, vnodes=32, slo_us=slo, batch=n, capacity=1 << 15, block_tokens=B,
                 route_prefix_blocks=1)
    p = Pair(w, max_instances=8, max_batch_tokens=1 << 20, max_touch=1 << 15, max_queue=1 << 14, choice_rule=5)
    for i in range(8):
        assert p.add(i) == 0
    rng = np.random.default_rng(9)
    starts = rng.integers(0, 32000, (400, B), dtype=np.uint32)
    pos = np.array([p.ora.prompt_keys(x)[1] for x in starts], np.uint64)
    c1 = p.ora.ring_owners(pos[:, 0].copy(), 0)
    for t in (1, 2):
        pick = np.concatenate([rng.choice(np.nonzero(c1 == i)[0], k) for i, k in enumerate(share) if k])
        rng.shuffle(pick)
        lens = rng.integers(B, 2 * B, n).astype(np.uint32)
        off = np.arange(n, dtype=np.uint64) * np.uint64(2 * B)
        tok = np.zeros((n, 2 * B), np.uint32)
        tok[:, :B] = starts[pick]
        p.route(tok.reshape(-1), off, lens, t)
        moved = p.rebalance()
        assert (moved > 0) == (slo > 1)
        p.commit()
    p.check_state(tag="end")
    p.gpu.close()
