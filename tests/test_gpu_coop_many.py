"""The cooperative kernel's form for more queries than the GPU holds at once (four
distance warps, more blocks per SM), which wide rows take: FP32 and 16-bit rows on
both sides of 32, 64, 128 and 256 chunks, plain and persistent, in both
verification modes, against the same queries in batches that are all resident.
Every row is summed by the same lanes in the same order: equal bit for bit."""
import numpy as np
import pytest

from helpers import workload_arrays
from paper_2605_02030_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(132, "f32"), (256, "f32"), (300, "f32"), (512, "f32"), (960, "f32"),
                                     (1028, "f32"), (520, "f16"), (960, "bf16"), (1100, "f16")])
def test_many_queries_equal_few(d, dtype):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    w, base, qs, p, _, _ = workload_arrays("mixture10k", 1500, 300, d=d, M=8, ef_construction=40)
    g = [U.build_graph(base, m, 8, 40, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    idx = U.Index(base, g[0], g[1], traverse_dtype=dtype)
    p = p.copy()
    p[::7], p[3::7], p[5::7] = 1.0, 2.0, 0.5
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    row = torch.arange(20 * sms, device="cuda") % len(qs)
    q, pd = torch.from_numpy(qs).cuda(), torch.from_numpy(p).cuda()
    qm, pm = q[row].contiguous(), pd[row].contiguous()
    for c in (dict(k=10, ef=150, width=1), dict(k=20, ef=140, width=2, mode="paper")):
        ref = idx.search(q, pd, query_threads=128, stats=True, **c)
        for threads in (0, 128):
            for persistent in (False, True):
                got = idx.search(qm, pm, query_threads=threads, persistent=persistent, stats=True, **c)
                assert torch.equal(got[0], ref[0][row]) and torch.equal(got[1], ref[1][row]), (c, threads)
                assert torch.equal(got[2][:, [1, 3, 5, 6, 7]], ref[2][row][:, [1, 3, 5, 6, 7]])
    assert idx.device_status() == 0
    idx.close()
