"""Exhaustive search where its split of the work changes: 4, 8 and 16 queries per
block (by the tiles per SM, on both sides of each line, for lists of up to 128 and
longer ones), lists shorter than k in some of a block's row groups, and one to many
slices.  Integer rows under L1 and L2: sums are exact, so that ids are equal to the
(S, id) order and distances to the rounded roots."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(70, 8), (300, 24), (1000, 8), (2100, 17)])
@pytest.mark.parametrize("k", [1, 20, 128, 129, 256])
def test_exact_across_the_split(n, d, k):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    rng = np.random.default_rng(n * 1000 + d + k)
    base = rng.integers(0, 30, (n, d)).astype(np.float32)
    level = {"nodes": np.arange(n, dtype=np.int32), "offsets": np.arange(n + 1, dtype=np.int64),
             "nbrs": np.arange(1, n + 1, dtype=np.int32) % n}
    idx = U.Index(base, {"num_levels": 1, "entry_point": 0, "max_degree0": 1, "max_degree": 1, "n": n,
                         "levels": [level]}, None)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-n // 128)
    x = torch.from_numpy(base).cuda().double()
    m = min(n, k)
    sizes = {3, 5, 8, 9}
    for line, per in ((2 * sms, 8), (2 * sms, 16), (14 * sms, 16)):
        at = -(-line // tiles) * per            # the first size past the line
        sizes |= {s for s in (at - per, at) if 0 < s <= 6000}
    most = max(sizes)
    qs = torch.from_numpy(rng.integers(0, 30, (most, d)).astype(np.float32)).cuda()
    p = torch.from_numpy(rng.choice(np.float32([1.0, 2.0]), most)).cuda()
    ref = torch.empty((most, m), dtype=torch.int64, device="cuda")
    dist = torch.empty((most, m), dtype=torch.float64, device="cuda")
    for s in range(0, most, 256):
        diff = (x[None] - qs[s:s + 256, None].double()).abs()
        S = torch.where(p[s:s + 256, None] == 1, diff.sum(-1), (diff * diff).sum(-1))
        key = (S.long() * n + torch.arange(n, device="cuda")).sort(dim=1).values[:, :m]
        ref[s:s + 256], dist[s:s + 256] = key % n, (key // n).double()
    dist = torch.where(p[:, None] == 1, dist, dist.sqrt()).float()
    for nq in sorted(sizes):
        ids, got = idx.exact(qs[:nq].contiguous(), p[:nq].contiguous(), k)
        assert torch.equal(ids[:, :m], ref[:nq]) and torch.equal(got[:, :m], dist[:nq]), nq
        assert (ids[:, m:] == -1).all() and torch.isinf(got[:, m:]).all()
    idx.close()
