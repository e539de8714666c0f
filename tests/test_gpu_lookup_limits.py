"""Index lookups that reach the limit of their bucket walk
(`test_loop_limit`): a lookup looks into that many buckets of its key's probe
order and no more, and one still open then ends the call in a sticky
DM_ERR_TIMEOUT.  Prompts of whole bucket groups (8 blocks) with the same home
bucket are routed and committed one after the other, so that the second group
lies in the second bucket of its order and each key of the third one in its
third."""

import numpy as np
import pytest

from oracle import oracle as O
from parity_harness import OUT_KEYS, lib_ready
from tracegen import workload

pytestmark = pytest.mark.gpu

B, SLOTS = 16, 256   # 32 buckets
CFG = workload("tiny", n_instances=4, vnodes=8, block_tokens=B, route_prefix_blocks=4, capacity=64, batch=64)


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


def bucket(j, home, key):
    """Bucket j of the probe order of a key with home bucket `home`."""
    if j == 0:
        return home
    if j == 1:
        b = O.fmix64(home ^ 0x5BD1E995A4C3B2E1) & (SLOTS - 8)
        return b if b != home else (home + 8) & (SLOTS - 1)
    return (O.fmix64(key) & (SLOTS - 8)) + (j - 2) * 8 & (SLOTS - 1)


class Sides:
    """An oracle and a scheduler with a limit, the same four instances."""

    def __init__(self, limit, rule, M):
        from paper_2602_06502_gb300.scheduler import Scheduler
        self.ora = O.Oracle(**O.config_from_workload(CFG, max_instances=M, max_batch_tokens=1 << 16), choice_rule=rule)
        self.gpu = Scheduler(block_tokens=B, route_prefix_blocks=4, vnodes=8, max_instances=M, capacity=64,
                             slo_us=CFG["slo_us"], cost_us=CFG["cost_us"], max_batch=64, max_batch_tokens=1 << 16,
                             max_touch_per_instance=64, index_slots_log2=8, max_queue=256, seed=CFG["seed"],
                             choice_rule=rule, test_loop_limit=limit)
        for i in range(4):
            assert self.ora.add_instance(i) == 0 and self.gpu.add_instance(i) == 0
        self.t = 0

    def info(self, tokens):
        """Home buckets of the prompt's groups, its keys and its two candidates."""
        keys, pos = self.ora.prompt_keys(tokens)
        keys = [int(k) for k in keys]
        c1 = int(self.ora.ring_owners(np.array([pos[0]], np.uint64), 0)[0])
        c2 = int(self.ora.ring_owners(np.array([pos[1]], np.uint64), 1)[0])
        return [k & (SLOTS - 8) for k in keys[::8]], keys, {c1, c2 if c2 != c1 else self.ora.next_live(c1)}, c1

    def route(self, prompts):
        """Routes a batch (every earlier request done by then) on the scheduler, and on the oracle for its outputs."""
        import torch
        self.t += 1_000_000
        lens = np.array([len(p) for p in prompts], np.uint32)
        off = (np.cumsum(lens) - lens).astype(np.uint64)
        tok = np.concatenate(prompts).astype(np.uint32)
        rc, want = self.ora.route_batch(tok, off, lens, self.t)
        assert rc == 0
        self.gpu.route(*[torch.from_numpy(x).cuda() for x in (tok.view(np.int32), off.view(np.int64),
                                                               lens.view(np.int32))], len(lens), len(tok), self.t)
        return want, self.gpu.results(len(lens))

    def commit(self):
        assert self.ora.commit() == 0
        self.gpu.commit()
        assert self.gpu.last_error() == 0


def _search(rng, blocks, s, ok):
    for _ in range(200_000):
        p = rng.integers(0, 32000, blocks * B, dtype=np.uint32)
        i = s.info(p)
        if ok(*i):
            return p, i
    raise AssertionError("no such prompt")


@pytest.mark.parametrize("limit", [0, 1, 2, 3])
def test_routing_lookup_limit(limit):
    from paper_2602_06502_gb300 import dualmap as D
    s = Sides(limit, 5, 4)   # rule 5: always the first candidate
    rng = np.random.default_rng(3)
    first, (h, _, _, c1) = _search(rng, 8, s, lambda *a: True)
    home, prompts = h[0], [first]
    taken = {bucket(0, home, 0), bucket(1, home, 0)}
    while len(prompts) < 3:
        prompts.append(_search(rng, 8, s, lambda g, keys, _, c: g[0] == home and c == c1 and
                               not taken & {bucket(2, home, k) for k in keys})[0])
    # prompt k is new and finds the first k buckets of its order full; then it is in bucket k
    for k, p in enumerate(prompts + prompts):
        want, got = s.route([p])
        if limit and k % 3 >= limit:
            assert s.gpu.last_error() == D.DM_ERR_TIMEOUT
            assert D.dm_commit_cache(s.gpu.h) == D.DM_ERR_TIMEOUT
            break
        assert s.gpu.last_error() == 0
        assert want["hit1"][0] == (8 * B if k >= 3 else 0)
        for f in OUT_KEYS:
            assert np.array_equal(got[f].astype(want[f].dtype), want[f]), (k, f)
        s.commit()
    assert k == (limit if limit in (1, 2) else 5)
    s.gpu.close()


@pytest.mark.parametrize("limit", [0, 1])
def test_cluster_probe_that_gives_up_inside_a_run(limit):
    """A resident prompt whose second group lies past the limit on an instance
    that is not its candidate: the cluster-wide probe finds a lower block
    missing and a higher one resident, and ends in the status."""
    from paper_2602_06502_gb300 import dualmap as D
    M = 512                     # 40 requests x 512 instances: a lane per pair
    s = Sides(limit, 6, M)      # rule 6: least loaded, so a lone request goes to instance 0
    rng = np.random.default_rng(5)

    def away(cands):
        return 0 not in cands

    prompt, (homes, _, _, _) = _search(
        rng, 40, s, lambda g, _, c, __: away(c) and len(set(g)) == 5 and bucket(1, g[1], 0) not in g)
    filler = _search(rng, 8, s, lambda g, _, c, __: g[0] == homes[1] and away(c))[0]
    others = [_search(rng, 1, s, lambda g, _, c, __: away(c))[0] for _ in range(39)]
    for p in (filler, prompt):
        want, _ = s.route([p])
        assert want["chosen"][0] == 0
        s.commit()
    want, got = s.route([prompt] + others)
    if limit:
        assert s.gpu.last_error() == D.DM_ERR_TIMEOUT
        assert D.dm_commit_cache(s.gpu.h) == D.DM_ERR_TIMEOUT
    else:
        assert s.gpu.last_error() == 0
        for k in OUT_KEYS:
            assert np.array_equal(got[k].astype(want[k].dtype), want[k]), k
    s.gpu.close()
