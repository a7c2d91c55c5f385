"""The cooperative kernel's form for more queries than the GPU holds at once, in which
the warps of a block share a step's rows: every number of links a warp can have (from
one to the 32 that it holds at once, and past them, where the form is not taken), one
to eight expansions a step, tables that are refilled, against the same queries in
batches that are all resident.  Who sums a row is left to timing; its lanes, their
order and the place of its key are not: equal bit for bit, on every run."""
import numpy as np
import pytest

from helpers import workload_arrays
from paper_2605_02030_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(250, "f32"), (400, "f32"), (960, "f32"), (500, "f16"), (960, "bf16")])
@pytest.mark.parametrize("M", [2, 16, 48])
def test_shared_steps(d, dtype, M):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    w, base, qs, p, _, _ = workload_arrays("mixture10k", 1500, 200, d=d, M=M, ef_construction=40)
    g = [U.build_graph(base, m, M, 40, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    idx = U.Index(base, g[0], g[1], traverse_dtype=dtype)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    row = torch.arange(14 * sms, device="cuda") % len(qs)
    q, pd = torch.from_numpy(qs).cuda(), torch.from_numpy(p).cuda()
    qm, pm = q[row].contiguous(), pd[row].contiguous()
    for c in (dict(ef=40, width=1), dict(ef=150, width=1), dict(ef=60, width=2), dict(ef=60, width=3),
              dict(ef=60, width=8)):
        small = int(np.ceil(np.log2(2 * (c["ef"] + c["width"] * 2 * M))))
        ref = idx.search(q, pd, k=10, query_threads=128, stats=True, **c)
        for bits in (0, small):
            for persistent in (False, True):
                got = idx.search(qm, pm, k=10, query_threads=128, persistent=persistent, hash_bits=bits,
                                 stats=True, **c)
                assert torch.equal(got[0], ref[0][row]) and torch.equal(got[1], ref[1][row]), (c, bits)
                assert torch.equal(got[2][:, [1, 3, 5, 6, 7]], ref[2][row][:, [1, 3, 5, 6, 7]]), (c, bits)
    assert idx.device_status() == 0
    idx.close()
