"""Algorithm 1 with batches larger than any candidate list: kappa up to INT_MAX
is one batch after the first K, as kappa = ef is, in both search kernels and in
the verification (the end of a batch is taken without forming i + kappa)."""
import numpy as np
import pytest

from helpers import workload_arrays

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

INT_MAX = 2 ** 31 - 1


def test_batches_past_the_list():
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import inputs as I
    from paper_2605_02030_gb300 import uhnsw as U
    w, base, qs, p, _, _ = workload_arrays("mixture10k", 1500, 60, d=48, M=8, ef_construction=40)
    g = [U.build_graph(base, m, 8, 40, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    idx = U.Index(base, g[0], g[1])
    q, pd = torch.from_numpy(qs).cuda(), torch.from_numpy(p).cuda()
    gen = torch.Generator().manual_seed(3)
    cand = torch.stack([torch.randperm(len(base), generator=gen)[:200] for _ in range(len(qs))]).int().cuda()
    for threads in (0, 32, 128):
        o = dict(k=10, ef=100, mode="paper", query_threads=threads, stats=True)
        ref = idx.search(q, pd, kappa=100, **o)
        for kappa in (INT_MAX, INT_MAX - 5):
            got = idx.search(q, pd, kappa=kappa, **o)
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(ref[:2], got[:2])), (threads, kappa)
            assert torch.equal(ref[2][:, 1], got[2][:, 1]), (threads, kappa)
    ref = idx.verify(q, pd, cand, 10, mode="paper", kappa=200, stats=True)
    got = idx.verify(q, pd, cand, 10, mode="paper", kappa=INT_MAX, stats=True)
    assert torch.equal(ref[0], got[0]) and torch.equal(ref[1], got[1])
    assert torch.equal(ref[2][:, 1], got[2][:, 1])
    assert idx.device_status() == 0
    idx.close()
