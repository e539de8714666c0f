"""The cluster-wide rules at the sizes where their kernels change (instances a
lane holds: 64, 128, 256, 512, then any number) and where a chunk's loads and
work leave 31 bits, bit for bit against the oracle."""

import pytest

from parity_harness import Pair, lib_ready, run_trace
from tracegen import Trace, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


@pytest.mark.parametrize("rule,live,M,batch,cost", [
    (7, 2, 2, 65, 1), (6, 64, 64, 129, 1), (8, 65, 70, 64, 1), (7, 128, 128, 63, 1), (8, 129, 256, 200, 1),
    (7, 300, 512, 97, 1), (6, 40, 513, 130, 1), (8, 520, 600, 70, 1),
    # cost x length past 31 bits in every, then in some requests
    (7, 9, 64, 130, 1 << 25), (8, 9, 64, 130, 1 << 21), (6, 130, 140, 130, 1 << 21)])
def test_cluster_rules_at_kernel_edges(rule, live, M, batch, cost):
    w = workload("tiny", n_instances=live, vnodes=8, cost_us=cost, slo_us=30_000 * cost, zipf_s=1.2, rho=1.2,
                 n_requests=4 * batch, batch=batch, capacity=4096, len_lo=64, len_hi=1500)
    p = Pair(w, max_instances=M, max_batch_tokens=1 << 19, max_touch=1 << 14, max_queue=1024, choice_rule=rule)
    run_trace(p, Trace(w))
    p.gpu.close()
