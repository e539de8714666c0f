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
