"""Exhaustive search with p outside (0, 2], which it takes (no range of p is checked):
the sum has a term per dimension and none beside them, also where a row ends in the
middle of a chunk of 16 dimensions.  S = sum |x - q|^p with FP32 terms of SFU
accuracy, 2e-5 as everywhere, and twice that for the root at |p| = 0.5.  At p = 0 every term is 1 and every sum equal, so that
the first k rows are returned, at distance d^(1/0) = +inf."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [8, 16, 24, 40])
@pytest.mark.parametrize("nq", [3, 7, 40, 3000])
def test_terms_of_the_row_alone(d, nq):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    n, k = 700, 5
    rng = np.random.default_rng(d)
    base = rng.standard_normal((n, d)).astype(np.float32)
    level = {"nodes": np.arange(n, dtype=np.int32), "offsets": np.arange(n + 1, dtype=np.int64),
             "nbrs": np.arange(1, n + 1, dtype=np.int32) % n}
    idx = U.Index(base, {"num_levels": 1, "entry_point": 0, "max_degree0": 1, "max_degree": 1, "n": n,
                         "levels": [level]}, None)
    q = torch.from_numpy(rng.standard_normal((nq, d)).astype(np.float32)).cuda()
    p = torch.tensor([-1.0, 0.0, -0.5, 3.0, 2.5, 0.7], device="cuda")[torch.arange(nq, device="cuda") % 6]
    ids, dist = idx.exact(q, p.contiguous(), k)
    x = torch.from_numpy(base).cuda().double()
    for s in range(0, nq, 500):
        pp = p[s:s + 500].double()[:, None]
        S = (x[None] - q[s:s + 500, None].double()).abs().pow(pp[..., None]).sum(-1)
        top = S.topk(k, largest=False).values.sort(dim=1).values
        zero = pp[:, 0] == 0
        got = dist[s:s + 500].double()
        assert (ids[s:s + 500][zero] == torch.arange(k, device="cuda")).all() and torch.isinf(got[zero]).all()
        assert torch.allclose(got[~zero], top.pow(1.0 / pp)[~zero], rtol=4e-5)
        own = S.gather(1, ids[s:s + 500])
        assert torch.allclose(own[~zero], top[~zero], rtol=4e-5)
    idx.close()
