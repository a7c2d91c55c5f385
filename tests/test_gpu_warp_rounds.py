"""The warp kernel's two forms (24 or 32 warps per SM) at the batch sizes where the
choice between them changes: one round of 24 warps, one of 32, two of 24, and one
query more of each, plain and persistent, against the block-per-query kernel.
Integer rows: ids and distances are equal bit for bit."""
import numpy as np
import pytest

from helpers import workload_arrays
from paper_2605_02030_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_batches_around_a_round_of_warps():
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    w, base, qs, p, _, _ = workload_arrays("sift1m", 2000, 500, d=60, M=8, ef_construction=30)
    g = [U.build_graph(base, m, 8, 30, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    idx = U.Index(base, g[0], g[1])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    most = 48 * sms + 1
    row = torch.arange(most, device="cuda") % len(qs)
    q, pd = torch.from_numpy(qs).cuda()[row].contiguous(), torch.from_numpy(p).cuda()[row].contiguous()
    ref = idx.search(q[:len(qs)], pd[:len(qs)], k=10, ef=40, query_threads=128)
    for nq in (24 * sms, 24 * sms + 1, 32 * sms, 32 * sms + 1, 48 * sms, most):
        for persistent in (False, True):
            got = idx.search(q[:nq], pd[:nq], k=10, ef=40, query_threads=32, persistent=persistent)
            assert torch.equal(got[0], ref[0][row[:nq]]) and torch.equal(got[1], ref[1][row[:nq]]), nq
    assert idx.device_status() == 0
    idx.close()
