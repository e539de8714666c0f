"""Instance changes at the sizes where an id's virtual nodes are sorted
another way: one node, and around 2,048, 4,096 and 8,192 nodes (shared memory
without and with more than its default limit, then global memory), bit for bit
against the oracle's rings, next-live order and routing."""

import numpy as np
import pytest

from parity_harness import Pair, lib_ready
from tracegen import Trace, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


@pytest.mark.parametrize("vnodes", [1, 33, 2048, 2049, 4096, 4097, 8192, 8193])
def test_rings_after_instance_changes(vnodes):
    from paper_2602_06502_gb300 import dualmap as D
    tr = Trace(workload("tiny", n_requests=40, batch=20, n_instances=4, vnodes=vnodes, capacity=4096))
    p = Pair(tr.cfg, max_instances=5, max_batch_tokens=1 << 18)

    def rings(tag):
        for f in (0, 1):
            vp, ow, _ = p.ora.ring(f)
            gv, go = D.dm_export_ring(p.gpu.h, f, len(vp) + 8)
            assert np.array_equal(gv, vp) and np.array_equal(go, ow), (tag, f)

    for i in (3, 0, 4, 1):
        assert p.add(i) == 0
        rings(f"add {i}")
    for b, change in enumerate((lambda: p.remove(4), lambda: p.add(2))):
        assert change() == 0
        rings(f"change {b}")
        s, e, off, lens, ntok = tr.batch_layout(b)
        p.route(tr.batch_tokens(b), off, lens, tr.batch_time(b), tag=f"batch {b}")
        p.commit()
    p.check_state(tag="end")
    p.gpu.close()
