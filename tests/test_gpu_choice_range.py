"""The choices where the loads leave the range that is decided in 32 bits
(2^31, 2^28 with d candidates): always below it, passing it within a batch,
and always above it, bit for bit against the oracle."""

import numpy as np
import pytest

from oracle import oracle as O
from parity_harness import Pair, lib_ready, run_trace
from tracegen import Trace, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


def _trace(cost, batch=520, **kw):
    return Trace(workload("tiny", n_requests=batch * 4, batch=batch, zipf_s=1.2, rho=1.3, slo_us=40_000 * cost,
                          cost_us=cost, len_lo=64, len_hi=600, prefix_lo=32, prefix_hi=300, **kw))


@pytest.mark.parametrize("rule", [0, 1, 2, 3, 4, 5])
@pytest.mark.parametrize("cost", [1, 1 << 14, 1 << 23, (1 << 32) - 1])
def test_pair_choice_ranges(rule, cost):
    tr = _trace(cost)
    p = Pair(tr.cfg, max_batch_tokens=1 << 20, choice_rule=rule)
    run_trace(p, tr)
    p.gpu.close()


def test_pair_choice_distinct_instances():
    tr = _trace(1, batch=700, n_instances=300, vnodes=4)   # windows whose requests mostly share no instance
    p = Pair(tr.cfg, max_batch_tokens=1 << 20)
    run_trace(p, tr)
    p.gpu.close()


@pytest.mark.parametrize("d", [1, 3, 4, 8])
@pytest.mark.parametrize("cost", [1, 1 << 11, 1 << 20])
def test_d_choice_ranges(d, cost):
    import torch
    from paper_2602_06502_gb300.scheduler import Scheduler
    tr = _trace(cost)
    w = tr.cfg
    M = w["n_instances"] + 2
    ora = O.Oracle(**O.config_from_workload(w, max_instances=M, max_batch_tokens=1 << 20, candidates=d))
    gpu = Scheduler(block_tokens=w["block_tokens"], route_prefix_blocks=w["route_prefix_blocks"], vnodes=w["vnodes"],
                    max_instances=M, capacity=w["capacity"], slo_us=w["slo_us"], cost_us=w["cost_us"],
                    max_batch=w["batch"], max_batch_tokens=1 << 20, seed=w["seed"], candidates=d)
    for i in range(w["n_instances"]):
        assert ora.add_instance(i) == 0 and gpu.add_instance(i) == 0
    for b in range(len(tr.batches)):
        s, e, off, lens, ntok = tr.batch_layout(b)
        tok = tr.batch_tokens(b)
        rc, want = ora.route_batch_d(d, tok, off, lens, tr.batch_time(b))
        assert rc == 0
        gpu.route_d(*[torch.from_numpy(x).cuda() for x in (tok.view(np.int32), off.view(np.int64),
                                                           lens.view(np.int32))], e - s, ntok, tr.batch_time(b))
        got = gpu.results_d(e - s)
        for k in ("cand", "hit", "ttft", "chosen", "switched"):
            assert np.array_equal(got[k].astype(want[k].dtype), want[k]), (b, k)
        assert ora.commit() == 0
        gpu.commit()
    assert gpu.last_error() == 0 and np.array_equal(gpu.loads(), ora.loads())
    gpu.close()


@pytest.mark.parametrize("rule,M", [(6, 64), (7, 64), (8, 64), (7, 128), (8, 250), (7, 400)])
@pytest.mark.parametrize("cost", [1 << 10, 1 << 14, 1 << 19])
def test_cluster_choice_ranges(rule, M, cost):
    # loads and work below 2^31 but no longer beside the list index, then past 2^31
    tr = _trace(cost, batch=130, n_instances=min(M, 40), vnodes=4)
    p = Pair(tr.cfg, max_instances=M, max_batch_tokens=1 << 20, max_touch=1 << 13, max_queue=1024, choice_rule=rule)
    run_trace(p, tr)
    p.gpu.close()
