"""The chained launches of a bucketed persistent search (one launch per beam
bucket, each starting on the slots the one before leaves): calls queued back to
back on one stream share their queue heads and output buffers, and work queued
behind a call reads all of its results."""
import numpy as np
import pytest

from helpers import workload_arrays
from paper_2605_02030_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(64, "f16"), (96, "f16"), (128, "f32"), (700, "bf16")])
def test_back_to_back_chains(d, dtype):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    w, base, qs, p, _, _ = workload_arrays("mixture10k", 3000, 4100, d=d, M=16, ef_construction=40)
    g = [U.build_graph(base, m, 16, 40, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    idx = U.Index(base, g[0], g[1], traverse_dtype=dtype)
    rng = np.random.default_rng(d)
    ef = torch.from_numpy(rng.choice([16, 64, 65, 128, 200, 400, 512], len(qs)).astype(np.int32)).cuda()
    k = torch.from_numpy(rng.integers(1, 11, len(qs)).astype(np.int32)).cuda()
    q, pd = torch.from_numpy(qs).cuda(), torch.from_numpy(p).cuda()
    for nq in (1, 5, 700, 4100):
        ref = idx.search(q[:nq], pd[:nq], k[:nq], ef[:nq], k_max=10, ef_max=512)
        back = torch.arange(nq - 1, -1, -1, device="cuda")
        qr, pr, kr, er = (x[:nq][back].contiguous() for x in (q, pd, k, ef))
        for graph in (False, True):
            out = (torch.empty((nq, 10), dtype=torch.int64, device="cuda"),
                   torch.empty((nq, 10), device="cuda"))
            got = []
            for a in ((q[:nq], pd[:nq], k[:nq], ef[:nq]), (qr, pr, kr, er)) * 3:
                out[0].fill_(-7)
                idx.search(*a, k_max=10, ef_max=512, persistent=True, use_graph=graph, out=out)
                got.append((out[0].clone(), out[1].clone()))
            torch.cuda.synchronize()
            for i, (a, b) in enumerate(got):
                r = (ref[0], ref[1]) if i % 2 == 0 else (ref[0][back], ref[1][back])
                # float rows: the kernels of a bucket may add a row by other lanes
                assert torch.equal(a < 0, r[0] < 0), (nq, graph, i)
                fin = a >= 0
                assert torch.allclose(b[fin], r[1][fin], rtol=2e-5), (nq, graph, i)
                assert (a == r[0]).float().mean() > 0.99, (nq, graph, i)
    assert idx.device_status() == 0
    idx.close()
