"""The verification kernel (a block per query: 2, 4 or 8 warps sum the candidate
rows and one keeps the list) at the edges of its steps: lists that end before,
at and after 16, 32 and 64 candidates, list lengths K around the merge's chunk
sizes, the batch sizes where the number of warps changes, rows that do and do
not fill a 128-dimension load, absent candidates, and every p form.

Sums of up to 300 FP32 terms by 8 lanes: the relative error is at most about
38 additions x 2^-24 + the SFU's 2^-21 per term, below the 2e-5 used everywhere."""
import numpy as np
import pytest

from helpers import workload_arrays

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def U():
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw
    return uhnsw


def _reference(base, q, p, cand, k):
    """FP64 distances of each query's k nearest valid candidates (inf past them)."""
    x = torch.from_numpy(base).cuda().double()[cand.long().clamp(min=0)]
    s = (x - q[:, None].double()).abs().pow(p[:, None, None].double()).sum(-1)
    s = torch.where(cand < 0, torch.inf, s)
    s = torch.nn.functional.pad(s, (0, max(0, k - s.shape[1])), value=torch.inf)
    return s.sort(dim=1).values[:, :k].pow(1.0 / p[:, None].double())


@pytest.mark.parametrize("d", [7, 128, 300])
@pytest.mark.parametrize("t,k", [(1, 1), (15, 4), (16, 16), (17, 1), (32, 31), (33, 33), (63, 64), (65, 10),
                                 (129, 65), (300, 129), (700, 512)])
def test_steps_and_warps(U, d, t, k):
    w, base, qs, p, _, _ = workload_arrays("mixture10k", 1200, 40, d=d, M=8)
    n = len(base)
    chain = {"num_levels": 1, "entry_point": 0, "max_degree0": 1, "max_degree": 1, "n": n,
             "levels": [{"nodes": np.arange(n, dtype=np.int32), "offsets": np.arange(n + 1, dtype=np.int64),
                         "nbrs": np.arange(1, n + 1, dtype=np.int32) % n}]}
    idx = U.Index(base, chain, None)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator().manual_seed(t * 1000 + k)
    p = p.copy()
    p[:5] = [0.5, 1.0, 1.5, 2.0, 0.2]
    cand = torch.stack([torch.randperm(n, generator=g)[:t] for _ in range(len(qs))]).int()
    cand[torch.rand(cand.shape, generator=g) < 0.1] = -1
    q, pp, cand = torch.from_numpy(qs).cuda(), torch.from_numpy(p).cuda(), cand.cuda()
    ref = _reference(base, q, pp, cand, k)
    few = idx.verify(q, pp, cand, k)
    assert torch.equal(torch.isinf(ref), torch.isinf(few[1]))
    fin = ~torch.isinf(ref)
    assert torch.equal(fin, few[0] >= 0)
    rel = ((few[1].double() - ref) / ref)[fin & (ref > 0)]
    assert rel.numel() == 0 or rel.abs().max() < 2e-5
    # the ids' own distances, and no id twice
    own = torch.stack([_reference(base, q[i:i + 1], pp[i:i + 1], few[0][i:i + 1].int(), k)[0]
                       for i in range(len(qs))])
    assert torch.allclose(own[fin], few[1].double().sort(dim=1).values[fin], rtol=2e-5)
    for row in few[0].cpu().tolist():
        row = [v for v in row if v >= 0]
        assert len(set(row)) == len(row)
    # more queries than 8 warps each are taken for: the same answers bit for bit
    r = torch.arange(3 * sms + 1, device="cuda") % len(qs)
    for mode in ("exact", "paper"):
        one = idx.verify(q, pp, cand, k, mode=mode, stats=True)
        many = idx.verify(q[r], pp[r], cand[r], k, mode=mode, stats=True)
        assert torch.equal(one[0][r], many[0]) and torch.equal(one[1][r], many[1])
        assert torch.equal(one[2][r][:, [1, 5]], many[2][:, [1, 5]])
    torch.cuda.synchronize()
    assert idx.device_status() == 0
    idx.close()
