"""Exhaustive search at the edges of its tiles: numbers of queries around the 4,
8 and 16 that share a block, rows around the 128 of a tile, k = 1, k past the
rows and the largest k, dimensions that do not fill a chunk of 16."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _index(base):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    n = len(base)
    level = {"nodes": np.arange(n, dtype=np.int32), "offsets": np.arange(n + 1, dtype=np.int64),
             "nbrs": (np.arange(1, n + 1, dtype=np.int32) % n)}
    g = {"num_levels": 1, "entry_point": 0, "max_degree0": 1, "max_degree": 1, "n": n,
         "levels": [level]}
    return U.Index(base, g, None)


@pytest.mark.parametrize("n,d", [(1, 3), (127, 16), (128, 17), (129, 40), (3001, 128)])
@pytest.mark.parametrize("k", [1, 33, 256])
def test_exact_at_tile_edges(n, d, k):
    rng = np.random.default_rng(n + d + k)
    base = rng.integers(0, 12, (n, d)).astype(np.float32)     # ties, and exact L1 / L2 sums
    idx = _index(base)
    for nq in (1, 4, 5, 8, 9, 17):
        qs = rng.integers(0, 12, (nq, d)).astype(np.float32)
        p = rng.choice(np.float32([0.5, 0.7, 1.0, 1.5, 2.0]), nq).astype(np.float32)
        ids, dist = idx.exact(torch.from_numpy(qs).cuda(), torch.from_numpy(p).cuda(), k)
        ids, dist = ids.cpu().numpy(), dist.cpu().numpy()
        m = min(n, k)
        for i in range(nq):
            S = (np.abs(base.astype(np.float64) - qs[i]) ** np.float64(p[i])).sum(1)
            order = np.lexsort((np.arange(n), S))[:m]
            assert (ids[i, m:] == -1).all() and np.isinf(dist[i, m:]).all()
            if p[i] in (1.0, 2.0):
                np.testing.assert_array_equal(ids[i, :m], order)
            # FP32 sums of up to 128 terms of SFU accuracy: 2e-5 as everywhere
            np.testing.assert_allclose(dist[i, :m], S[order] ** (1.0 / np.float64(p[i])), rtol=2e-5)
            np.testing.assert_allclose(S[ids[i, :m]], S[order], rtol=2e-5 * 2)
            assert len(set(ids[i, :m].tolist())) == m
    idx.close()
