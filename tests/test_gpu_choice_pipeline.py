"""The choice pipeline at the edges of its windows (32 requests) and chunks
(256, or 128 for more than four candidates), bit for bit against the oracle:
decisions, TTFTs, loads, queues, and the records' order in the caches."""

import numpy as np
import pytest

from oracle import oracle as O
from parity_harness import Pair, lib_ready, run_trace
from tracegen import Trace, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


def _trace(batch, batches=4):
    # few instances and hot prefixes: long chains of requests on one pair
    return Trace(workload("tiny", n_requests=batch * batches, batch=batch, zipf_s=1.2, rho=1.3, slo_us=40_000,
                          len_lo=64, len_hi=600, prefix_lo=32, prefix_hi=300))


@pytest.mark.parametrize("batch,rule", [(1, 0), (31, 0), (33, 4), (255, 0), (256, 3), (257, 0), (512, 0), (1025, 2)])
def test_pair_choice_window_and_chunk_edges(batch, rule):
    tr = _trace(batch)
    p = Pair(tr.cfg, max_batch_tokens=1 << 20, choice_rule=rule)
    run_trace(p, tr)
    p.gpu.close()


@pytest.mark.parametrize("batch,d", [(1, 5), (32, 2), (127, 8), (128, 6), (129, 7), (256, 4), (257, 3), (385, 5)])
def test_d_choice_window_and_chunk_edges(batch, d):
    import torch
    from paper_2602_06502_gb300 import dualmap as D
    from paper_2602_06502_gb300.scheduler import Scheduler
    tr = _trace(batch)
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
    for i in range(M):
        for a, g in zip(ora.queue(i), D.dm_export_queue(gpu.h, i)):
            assert np.array_equal(a, g), i
        ok, os_ = ora.cache(i)
        gk, gs = D.dm_export_cache(gpu.h, i)
        o, q = np.lexsort((ok, os_)), np.lexsort((gk, gs))
        assert np.array_equal(ok[o], gk[q]) and np.array_equal(os_[o], gs[q]), i
    gpu.close()
