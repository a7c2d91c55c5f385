"""The chained launches of a bucketed persistent search against the plain launch, bit
for bit.  The rows hold small integers, so that base sums are exact whatever lanes add
them, and the L_p sums are added by the same lanes in every kernel: ids and distances
are equal although the buckets' launches overlap, over calls queued back to back on one
stream and on two, replayed as graphs too."""
import numpy as np
import pytest

from helpers import workload_arrays
from paper_2605_02030_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(96, "f16"), (128, "f32"), (300, "f32"), (700, "bf16")])
def test_chains_equal_the_plain_launch(d, dtype):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    w, base, qs, p, _, _ = workload_arrays("sift1m", 2500, 700, d=d, M=16, ef_construction=40)
    most = 255.0 if d <= 128 else 150.0          # L2 sums below 2^24
    base, qs = (np.ascontiguousarray(np.minimum(x, most), np.float32) for x in (base, qs))
    p = p.copy()
    p[::5], p[1::5], p[2::5] = 1.0, 2.0, 0.5
    g = [U.build_graph(base, m, 16, 40, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    idx = U.Index(base, g[0], g[1], traverse_dtype=dtype)
    rng = np.random.default_rng(d)
    row = torch.from_numpy(rng.integers(0, len(qs), 4100)).cuda()
    q, pd = torch.from_numpy(qs).cuda()[row].contiguous(), torch.from_numpy(p).cuda()[row].contiguous()
    ef = torch.from_numpy(rng.choice([16, 64, 65, 128, 200, 400, 512], 4100).astype(np.int32)).cuda()
    k = torch.from_numpy(rng.integers(1, 11, 4100).astype(np.int32)).cuda()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for nq in (1, 5, 700, 4100):
        a = (q[:nq], pd[:nq], k[:nq], ef[:nq])
        ref = idx.search(*a, k_max=10, ef_max=512)
        torch.cuda.synchronize()
        for graph in (False, True):
            outs = [(torch.empty((nq, 10), dtype=torch.int64, device="cuda"),
                     torch.empty((nq, 10), device="cuda")) for _ in streams]
            for turn in range(4):
                for o in outs:
                    o[0].fill_(-7)
                torch.cuda.synchronize()
                for _ in range(3):
                    for s, o in zip(streams, outs):
                        idx.search(*a, k_max=10, ef_max=512, persistent=True, use_graph=graph, out=o,
                                   stream=s)
                torch.cuda.synchronize()
                for o in outs:
                    assert torch.equal(o[0], ref[0]) and torch.equal(o[1], ref[1]), (nq, graph, turn)
    assert idx.device_status() == 0
    idx.close()
