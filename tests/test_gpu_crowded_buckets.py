"""Leading runs in crowded indices: prompts that leave shared prefixes at every
block of a bucket group, an index as full as it gets, runs that end at the
edges of groups (8 blocks), words (32) and segments (64), and repeated prompts,
bit for bit against the oracle (two candidates, d candidates, moved requests'
fresh probes)."""

import numpy as np
import pytest

from oracle import oracle as O
from parity_harness import Pair, lib_ready
from tracegen import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


def _batches(seed, B, n, nb, longest):
    rng = np.random.default_rng(seed)
    prefixes = [rng.integers(0, 1000, longest * B, dtype=np.uint32) for _ in range(5)]
    edges = [1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128, 129]
    old, out = [], []
    for _ in range(nb):
        prompts = []
        for k in range(n):
            if old and k % 5 == 0:   # an earlier prompt again, or with a few blocks more
                p = old[rng.integers(len(old))]
                p = np.concatenate([p, rng.integers(0, 1000, int(rng.integers(0, 3)) * B, dtype=np.uint32)])
            else:
                keep = int(rng.choice(edges) if k % 2 else rng.integers(1, longest))
                own = int(rng.integers(0, 40)) * B + int(rng.integers(0, B))
                p = np.concatenate([prefixes[rng.integers(5)][:min(keep, longest) * B],
                                    rng.integers(0, 1000, own, dtype=np.uint32)])
            prompts.append(p[:4 * longest * B])
        old = (old + prompts)[-150:]
        lens = np.array([len(p) for p in prompts], np.uint32)
        room = (lens.astype(np.uint64) + 3) // 4 * 4
        off = np.cumsum(room) - room
        tok = np.zeros(int(room.sum()), np.uint32)
        for p, o in zip(prompts, off):
            tok[int(o):int(o) + len(p)] = p
        out.append((tok, off.astype(np.uint64), lens))
    return out


def _cfg(B, n, **kw):
    return workload("tiny", n_instances=4, vnodes=16, block_tokens=B, route_prefix_blocks=4, batch=n,
                    slo_us=20_000_000, **kw)


@pytest.mark.parametrize("B,longest,capacity,rebalance,flags", [
    (4, 140, 6000, False, 0), (16, 66, 3000, True, 0), (16, 140, 12000, True, 2), (64, 34, 2000, False, 0)])
def test_crowded_pair(B, longest, capacity, rebalance, flags):
    n = 120
    w = _cfg(B, n, capacity=capacity)
    p = Pair(w, max_instances=5, max_batch_tokens=1 << 21, max_touch=n * (longest * 4 + 1), rebalance_flags=flags,
             rebalance_key_blocks=1 << 18 if flags else 0)
    for i in range(4):
        assert p.add(i) == 0
    for b, (tok, off, lens) in enumerate(_batches(7 * B + longest, B, n, 10, longest)):
        p.route(tok, off, lens, b * 400_000, tag=f"batch {b}")
        if rebalance:
            p.rebalance(tag=f"batch {b}")
        p.commit()
    p.check_state()
    assert p.hit_tokens > 0
    p.gpu.close()


@pytest.mark.parametrize("d", [1, 3, 4])
def test_crowded_d(d):
    import torch
    from paper_2602_06502_gb300.scheduler import Scheduler
    B, n, longest = 16, 100, 140
    w = _cfg(B, n, capacity=5000)
    kw = dict(max_instances=5, max_batch_tokens=1 << 21)
    ora = O.Oracle(**O.config_from_workload(w, candidates=d, **kw))
    gpu = Scheduler(block_tokens=B, route_prefix_blocks=4, vnodes=w["vnodes"], capacity=w["capacity"],
                    slo_us=w["slo_us"], cost_us=w["cost_us"], max_batch=n, max_touch_per_instance=n * (longest * 4 + 1),
                    seed=w["seed"], candidates=d, **kw)
    for i in range(4):
        assert ora.add_instance(i) == 0 and gpu.add_instance(i) == 0
    for b, (tok, off, lens) in enumerate(_batches(d, B, n, 8, longest)):
        rc, want = ora.route_batch_d(d, tok, off, lens, b * 400_000)
        assert rc == 0
        gpu.route_d(*[torch.from_numpy(x).cuda() for x in (tok.view(np.int32), off.view(np.int64),
                                                           lens.view(np.int32))], n, len(tok), b * 400_000)
        got = gpu.results_d(n)
        for k in ("cand", "hit", "ttft", "chosen", "switched"):
            assert np.array_equal(got[k].astype(want[k].dtype), want[k]), (b, k)
        assert ora.commit() == 0
        gpu.commit()
    assert gpu.last_error() == 0
    gpu.close()
