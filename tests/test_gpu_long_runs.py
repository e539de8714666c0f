"""Cached runs that go on past a prompt's head (24 segments of 64 blocks):
runs ending at the head's edge, at and inside the segments after it, past a
round of 128 tail segments, and covering the whole prompt, bit for bit
against the oracle."""

import numpy as np
import pytest

from parity_harness import Pair, lib_ready
from tracegen import workload

pytestmark = pytest.mark.gpu

HEAD, ROUND = 24 * 64, 128 * 64   # blocks


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


@pytest.mark.parametrize("B,adapt", [(4, None), (16, None),
                                     (4, dict(adapt_step_blocks=64, adapt_max_blocks=2048, adapt_window=2))])
def test_run_past_the_head(B, adapt):
    edges = [HEAD - 1, HEAD, HEAD + 1, HEAD + 63, HEAD + 64, HEAD + 65, HEAD + 5 * 64 + 7, HEAD + ROUND - 1,
             HEAD + ROUND, HEAD + ROUND + 1, HEAD + ROUND + 64, HEAD + ROUND + 77]
    if B == 16:
        edges = edges[:7]
    total = edges[-1] + 130
    w = workload("tiny", n_instances=3, block_tokens=B, vnodes=16, capacity=1 << 17, batch=len(edges) + 4)
    p = Pair(w, max_batch_tokens=(len(edges) + 4) * (total + 4) * B, max_touch=1 << 18, adapt=adapt)
    for i in range(3):
        p.add(i)
    rng = np.random.default_rng(11)
    docs = [rng.integers(0, 32000, total * B, dtype=np.uint32) for _ in range(2)]

    def batch(prompts, t):
        lens = np.array([len(x) for x in prompts], np.uint32)
        room = (lens.astype(np.int64) + 3) // 4 * 4
        off = (np.cumsum(room) - room).astype(np.uint64)
        tok = np.zeros(int(room.sum()), np.uint32)
        for o, x in zip(off, prompts):
            tok[int(o):int(o) + len(x)] = x
        p.route(tok, off, lens, t, tag=f"t={t}")
        p.commit()

    # the documents up to each edge are cached one after the other, longest
    # last; each is then asked for again whole, cut inside, and with a new end
    for k, e in enumerate(edges):
        doc = docs[k % 2]
        batch([doc[:e * B]], 10 * k + 1)
        tail = rng.integers(0, 32000, 70 * B + 3, dtype=np.uint32)
        batch([doc[:e * B], np.concatenate([doc[:e * B], tail]), doc[:(e - 2) * B + 1], doc], 10 * k + 2)
    batch([docs[k % 2][:e * B + 1] for k, e in enumerate(edges)], 10_000)
    p.check_state(tag="end")
    assert p.hit_tokens > 0
    p.gpu.close()


def test_many_runs_past_the_head_at_once():
    """Runs past the head in every request of a batch, settled by whichever
    warp completes them: candidates, first misses and carries change with every
    batch in every place, so a value left from the batch before would show."""
    B, n, per = 4, 48, 12
    total = HEAD + 3 * ROUND // 4
    w = workload("tiny", n_instances=7, block_tokens=B, vnodes=16, capacity=1 << 17, batch=n)
    p = Pair(w, max_batch_tokens=n * (total + 8) * B, max_touch=n * total, max_queue=4096)
    for i in range(7):
        p.add(i)
    rng = np.random.default_rng(23)
    docs = [rng.integers(0, 32000, total * B, dtype=np.uint32) for _ in range(per)]
    for t in range(8):
        prompts = []
        for _ in range(n if t else per):
            k = int(rng.integers(per))
            cut = int(rng.integers(HEAD - 64, total + 1))
            own = rng.integers(0, 32000, int(rng.integers(0, 3 * 64)) * B, dtype=np.uint32)
            prompts.append(np.concatenate([docs[k][:cut * B], own])[:total * B])
        lens = np.array([len(x) for x in prompts], np.uint32)
        off = (np.cumsum(lens) - lens).astype(np.uint64)
        p.route(np.concatenate(prompts), off, lens, 100_000_000 * (t + 1), tag=f"batch {t}")
        p.commit()
    p.check_state(tag="end")
    assert p.hit_tokens > 0
    p.gpu.close()
