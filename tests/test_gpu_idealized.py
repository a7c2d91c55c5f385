"""Idealized recall where the two searches behind it (the top K and the top t_max)
want different numbers of row slices: few queries, a small K, the largest t_max
and enough rows that the number of tiles bounds neither.  The counts are those of
the two exhaustive answers taken one by one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [1, 64, 96, 500])
@pytest.mark.parametrize("K,t_max", [(1, 256), (10, 256), (100, 256), (7, 33)])
def test_few_queries_and_many_rows(nq, K, t_max):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    n, d = 70_000, 8
    rng = np.random.default_rng(11)
    base = rng.standard_normal((n, d)).astype(np.float32)
    level = {"nodes": np.arange(n, dtype=np.int32), "offsets": np.arange(n + 1, dtype=np.int64),
             "nbrs": np.arange(1, n + 1, dtype=np.int32) % n}
    chain = {"num_levels": 1, "entry_point": 0, "max_degree0": 1, "max_degree": 1, "n": n,
             "levels": [level]}
    idx = U.Index(base, chain, None)
    q = torch.from_numpy(rng.standard_normal((nq, d)).astype(np.float32)).cuda()
    p = torch.from_numpy(rng.choice(np.float32([0.6, 1.0, 1.3, 1.7]), nq)).cuda()
    got = idx.idealized_recall(q, p, K, t_max)
    top_k = idx.exact(q, p, K)[0]
    top_t = idx.exact(q, torch.where(p <= 1.4, 1.0, 2.0).float(), t_max)[0]
    hit = (top_t[:, :, None] == top_k[:, None, :]).any(-1)
    assert torch.equal(got, hit.cumsum(1).to(got.dtype))
    idx.close()
