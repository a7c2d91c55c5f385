"""The root S^(1/p) of a returned distance, for p from the smallest positive FP32
number to 2.  The query is 0 and row m holds m ones, so that S = m exactly for
every p (|1|^p = 2^0 and |0|^p = 0) and only the root is left.

The root is within 2^-44 of the exact value before it is rounded to FP32, so it
is the rounded FP64 value or, where that lies within 2^-44 of the middle of two
FP32 numbers, the other one: one unit at most.  A root past FP32's range is
+inf, and S = 1 and S = 0 give 1 and 0 for every p."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_roots_of_whole_sums():
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    d = 1024
    ones = np.unique(np.concatenate([np.arange(260), np.linspace(260, d, 252).astype(int)]))
    base = (np.arange(d)[None] < ones[:, None]).astype(np.float32)
    n = len(base)
    chain = {"num_levels": 1, "entry_point": 0, "max_degree0": 1, "max_degree": 1, "n": n,
             "levels": [{"nodes": np.arange(n, dtype=np.int32), "offsets": np.arange(n + 1, dtype=np.int64),
                         "nbrs": np.arange(1, n + 1, dtype=np.int32) % n}]}
    idx = U.Index(base, chain, None)
    rng = np.random.default_rng(7)
    p = np.concatenate([[1.4e-45, 1e-44, 1e-39, 1.17e-38, 1.18e-38, 1e-30, 7.8e-31, 7.9e-31, 1e-20, 0.5, 1.0,
                         1.5, 2.0], 10.0 ** rng.uniform(-3, np.log10(2.0), 300)]).astype(np.float32)
    assert (p > 0).all() and (p <= 2).all()
    q = torch.zeros((len(p), d), device="cuda")
    cand = torch.arange(n, dtype=torch.int32, device="cuda").repeat(len(p), 1)
    ids, dist, st = idx.verify(q, torch.from_numpy(p).cuda(), cand, n, stats=True)
    ids, dist = ids.cpu().numpy(), dist.cpu().numpy()
    assert (st[:, 5] == 0).all() and (ids == np.arange(n)).all()
    with np.errstate(over="ignore", divide="ignore"):
        exact = (ones.astype(np.float64)[None] ** (1.0 / p.astype(np.float64)[:, None])).astype(np.float32)
    assert (np.isinf(dist) == np.isinf(exact)).all()
    fin = np.isfinite(exact)
    assert (np.abs(dist[fin] - exact[fin]) <= np.spacing(exact[fin])).all()
    assert (dist[:, ones == 1] == 1).all() and (dist[:, ones == 0] == 0).all()
    idx.close()
