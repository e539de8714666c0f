"""Commits in which more instances are over capacity than the eviction kernel
has clusters, so that clusters take several each and some start while others
have finished: every cluster must deal out the same list.  Caches bit for bit
against the oracle after every batch."""

import pytest

from parity_harness import Pair, lib_ready, run_trace
from tracegen import Trace, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


@pytest.mark.parametrize("live,capacity,batch", [(700, 24, 4000), (150, 60, 1200)])
def test_most_instances_over_capacity(live, capacity, batch):
    w = workload("tiny", n_instances=live, vnodes=8, capacity=capacity, n_requests=5 * batch, batch=batch, len_lo=128,
                 len_hi=700, n_prefix=3 * live, zipf_s=0.3, prefix_lo=32, prefix_hi=300)
    p = Pair(w, max_instances=live, max_batch_tokens=1 << 22, max_touch=1 << 13, max_queue=1024, choice_rule=2)
    full = []

    def commit():
        Pair.commit(p)
        full.append(sum(len(p.ora.cache(i)[0]) == capacity for i in range(live)))

    p.commit = commit
    run_trace(p, Trace(w), state_every=1)
    assert full[0] > live // 2 and full[-1] > 0.9 * live, full
    p.gpu.close()
