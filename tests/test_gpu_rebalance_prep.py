"""Commits after a rebalance that moved requests of the batch: the records of
every instance are laid out again in arrival order, at batch sizes around the
layout's windows (32 requests), passes (256) and groups of passes (1,024), bit
for bit against the oracle."""

import pytest

from parity_harness import Pair, lib_ready, run_trace
from tracegen import Trace, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


@pytest.mark.parametrize("live,batch", [(8, 33), (16, 257), (12, 1025), (300, 2100), (511, 1500), (512, 1500)])
def test_commit_after_moves(live, batch):
    # few virtual nodes: some instances own many prefixes, and a request's other candidate may be far less loaded
    w = workload("tiny", n_instances=live, vnodes=2, slo_us=100_000_000, n_prefix=60, zipf_s=1.2, rho=1.0,
                 n_requests=5 * batch, batch=batch, capacity=2048, len_lo=64, len_hi=1200, prefix_lo=64,
                 prefix_hi=1024)
    p = Pair(w, max_instances=live + 1, max_batch_tokens=1 << 22, max_touch=1 << 17, max_queue=1 << 13)
    run_trace(p, Trace(w), rebalance=True)
    assert p.n_migrations > 0
    p.gpu.close()
