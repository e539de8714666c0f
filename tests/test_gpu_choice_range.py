"""The choices where the loads leave the range that is decided in 32 bits:
always below it, passing it within a batch, and always above it, bit for bit
against the oracle.  A chunk of requests is decided in 32 bits while a bound on
every load it can reach stays below 2^30 (2^28 with d candidates; 2^31, or
2^31 less the bits of the list index, above the smallest load for the
cluster-wide rules); the bound is worked out here from the oracle's loads, and
a case states on which sides its chunks lie (empty: either)."""

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


def batch_work(ora, W, chosen, seq0):
    """Each request's work on the instance that got it, and the loads before the batch."""
    work, W = [0] * len(chosen), [int(x) for x in W]
    for i in set(int(c) for c in chosen):
        for q, w, _ in zip(*ora.queue(i)):
            if q >= seq0:
                work[int(q) - seq0] = int(w)
    for c, w in zip(chosen, work):
        W[int(c)] -= w
    return work, W


def bounded_chunks(W, most, chunk, limit):
    """Per chunk of the pair and d choices: 'n' where the bound stays below limit, else 'w' (most: each request's
    largest work)."""
    bound, out = max(min(w, limit) for w in W), ""
    for c in range(0, len(most), chunk):
        units = sum((min(int(x), limit) + 1023) >> 10 for x in most[c:c + chunk])
        bound = min(bound + (units << 10), limit)
        out += "n" if bound < limit else "w"
    return out


def cluster_chunks(W, chosen, work, full, M, live):
    """Per chunk of the cluster-wide choice: 'p' packed with the list index, 'n' in 31 bits, 'w' in 64 (full: each
    request's cost x length)."""
    chunk, bits = (64 if M <= 256 else 32), (6 if M <= 64 else 7 if M <= 128 else 8 if M <= 256 else 9)
    out = ""
    for c in range(0, len(full), chunk):
        loads, added = [W[i] for i in range(live)], sum(full[c:c + chunk])
        reach = max(loads) - min(loads) + added
        wide = max(full[c:c + chunk]) >= 1 << 31 or reach >= 1 << 31
        out += "w" if wide else "p" if reach < (1 << 31) >> bits else "n"
        for k in range(c, min(c + chunk, len(full))):
            W[int(chosen[k])] += work[k]
    return out


class Watched(Pair):
    """A pair that notes the sides of every batch's chunks."""

    def __init__(self, w, choice_rule=0, **kw):
        super().__init__(w, choice_rule=choice_rule, **kw)
        self.rule, self.seq, self.sides = choice_rule, 0, []

    def route(self, tok, off, lens, t_batch, tag=""):
        want = super().route(tok, off, lens, t_batch, tag)
        cost = int(self.w["cost_us"])
        work, W = batch_work(self.ora, self.ora.loads(), want["chosen"], self.seq)
        if self.rule < 6:
            most = [cost * (int(n) - min(int(a), int(b))) for n, a, b in zip(lens, want["hit1"], want["hit2"])]
            self.sides.append(bounded_chunks(W, most, 256, 1 << 30))
        else:
            self.sides.append(cluster_chunks(W, want["chosen"], work, [cost * int(n) for n in lens], self.M,
                                             self.w["n_instances"]))
        self.seq += len(lens)
        return want


@pytest.mark.parametrize("rule", [0, 1, 2, 3, 4, 5])
@pytest.mark.parametrize("cost,sides", [(1, "n"), (1 << 13, "nw"), (1 << 14, ""), (1 << 23, "w"),
                                        ((1 << 32) - 1, "w")])
def test_pair_choice_ranges(rule, cost, sides):
    tr = _trace(cost)
    p = Watched(tr.cfg, max_batch_tokens=1 << 20, choice_rule=rule)
    run_trace(p, tr)
    assert not sides or max((set(x) for x in p.sides), key=len) == set(sides), p.sides
    p.gpu.close()


def test_pair_choice_distinct_instances():
    tr = _trace(1, batch=700, n_instances=300, vnodes=4)   # windows whose requests mostly share no instance
    p = Pair(tr.cfg, max_batch_tokens=1 << 20)
    run_trace(p, tr)
    p.gpu.close()


@pytest.mark.parametrize("d", [1, 3, 4, 8])
@pytest.mark.parametrize("cost,sides", [(1, "n"), (1 << 11, "nw"), (1 << 20, "w")])
def test_d_choice_ranges(d, cost, sides):
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
    seq, seen = 0, []
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
        most = [cost * (int(n) - int(h)) for n, h in zip(lens, want["hit"].min(axis=1))]
        seen.append(bounded_chunks(batch_work(ora, ora.loads(), want["chosen"], seq)[1], most, 256 if d <= 4 else 128,
                                   1 << 28))
        seq += e - s
        assert ora.commit() == 0
        gpu.commit()
    assert max((set(x) for x in seen), key=len) == set(sides), seen
    assert gpu.last_error() == 0 and np.array_equal(gpu.loads(), ora.loads())
    gpu.close()


@pytest.mark.parametrize("rule,M", [(6, 64), (7, 64), (8, 64), (7, 128), (8, 250), (7, 400)])
@pytest.mark.parametrize("cost,sides", [(1 << 8, "p"), (1 << 10, ""), (1 << 12, "np"), (1 << 14, ""), (1 << 19, "nw")])
def test_cluster_choice_ranges(rule, M, cost, sides):
    # beside the list index, loads and work below 2^31 but no longer beside it, then past 2^31
    tr = _trace(cost, batch=130, n_instances=min(M, 40), vnodes=4)
    p = Watched(tr.cfg, max_instances=M, max_batch_tokens=1 << 20, max_touch=1 << 13, max_queue=1024, choice_rule=rule)
    run_trace(p, tr)
    assert not sides or max((set(x) for x in p.sides), key=len) == set(sides), p.sides
    p.gpu.close()
