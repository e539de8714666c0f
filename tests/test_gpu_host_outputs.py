"""Host-memory routing with outputs in pinned memory (written by one kernel), in
pageable memory (copied), and in a mix, at the edges of the kernel's blocks:
the same decisions as the oracle's."""

import numpy as np
import pytest

from parity_harness import OUT_KEYS, Pair, lib_ready
from tracegen import Trace, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


@pytest.mark.parametrize("batch", [1, 127, 128, 129, 700])
@pytest.mark.parametrize("kind", ["pinned", "pageable", "mixed", "offset"])
def test_host_outputs(batch, kind):
    import torch
    from paper_2602_06502_gb300 import dualmap as D
    from paper_2602_06502_gb300.scheduler import OUT_FIELDS
    tr = Trace(workload("tiny", n_requests=3 * batch, batch=batch, len_lo=64, len_hi=400, prefix_lo=32, prefix_hi=200))
    p = Pair(tr.cfg, max_batch_tokens=1 << 20)
    for i in range(tr.cfg["n_instances"]):
        assert p.add(i) == 0
    out = {}
    for j, (name, t) in enumerate(OUT_FIELDS):
        x = torch.full((batch + 1,), 77, dtype=t)
        if kind in ("pinned", "offset") or (kind == "mixed" and j != 5):
            x = x.pin_memory()
        out[name] = x[1:] if kind == "offset" else x[:batch]
    for b in range(len(tr.batches)):
        s, e, off, lens, ntok = tr.batch_layout(b)
        tok = tr.batch_tokens(b)
        rc, want = p.ora.route_batch(tok, off, lens, tr.batch_time(b))
        assert rc == 0
        t = [torch.from_numpy(np.ascontiguousarray(x)).pin_memory() for x in
             (tok.view(np.int32), off.view(np.int64), lens.view(np.int32))]
        bt = D.make_batch(*t, e - s, len(tok), tr.batch_time(b))
        assert D.dm_route_batch_host(p.gpu.h, bt, D.make_out(*[out[k] for k, _ in OUT_FIELDS])) == 0
        for k in OUT_KEYS:
            assert np.array_equal(out[k][:e - s].numpy().astype(want[k].dtype), want[k]), (b, k)
        p.commit()
    p.check_loads()
    p.gpu.close()
