"""The cooperative kernel (one query per block: 2, 4 or 8 warps sum its rows and
one keeps its beam) against the warp-per-query kernel.  Both sum every row with
the same lanes in the same order and merge by the same strict order, so ids and
distances must be equal bit for bit, on float data too: at the batch sizes
where the number of warps per query changes, for rows that do and do not fill
their team, for beams around the merge's chunk sizes (32, 64, 128), for k = 1
and k = ef, in both verification modes, and with several expansions per step."""
import numpy as np
import pytest

from helpers import workload_arrays
from paper_2605_02030_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def U():
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw
    return uhnsw


# d, dtype, M: team shapes 8x1, 8x2 (partly filled), 4x3, 8x2, 32x2, 32x4
SHAPES = [(17, "f32", 8), (100, "f16", 16), (96, "f16", 32), (128, "bf16", 16), (200, "f32", 16),
          (960, "bf16", 8)]


@pytest.mark.parametrize("d,dtype,M", SHAPES)
def test_cooperative_kernel_equals_the_warp_kernel(U, d, dtype, M):
    w, base, qs, p, _, _ = workload_arrays("mixture10k", 2500, 700, d=d, M=M, ef_construction=48)
    g = [U.build_graph(base, m, M, 48, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    idx = U.Index(base, g[0], g[1], traverse_dtype=dtype)
    p = p.copy()
    p[::7], p[3::7], p[5::7] = 1.0, 2.0, 0.5
    q, pd = torch.from_numpy(qs).cuda(), torch.from_numpy(p).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(1)
    kq = torch.from_numpy(rng.integers(1, 40, len(qs)).astype(np.int32)).cuda()
    eq = torch.from_numpy(rng.integers(1, 150, len(qs)).astype(np.int32)).cuda()
    cases = [dict(k=10, ef=64, width=1), dict(k=1, ef=1, width=1), dict(k=33, ef=33, width=2),
             dict(k=10, ef=65, width=3, mode="paper"), dict(k=20, ef=129, width=1, mode="paper"),
             dict(k=5, ef=32, width=8), dict(k=kq, ef=eq, width=2, k_max=40, ef_max=160),
             dict(k=kq, ef=eq, width=1, k_max=40, ef_max=160, persistent=True)]
    for nq in (1, sms, sms + 1, 4 * sms + 1, 700):
        for c in cases:
            c = {a: (b[:nq] if torch.is_tensor(b) else b) for a, b in c.items()}
            ref = idx.search(q[:nq], pd[:nq], query_threads=32, stats=True, **c)
            got = idx.search(q[:nq], pd[:nq], stats=True, **c)
            torch.cuda.synchronize()
            what = f"nq={nq} {c}"
            assert torch.equal(ref[0], got[0]) and torch.equal(ref[1], got[1]), what
            # expansions, adjacency rows and verified candidates are the same search's
            assert torch.equal(ref[2][:, [1, 3, 5, 6, 7]], got[2][:, [1, 3, 5, 6, 7]]), what
    assert idx.device_status() == 0
    idx.close()


def test_table_refills_change_no_result(U):
    """A visited table of the smallest allowed size is refilled many times."""
    w, base, qs, p, _, _ = workload_arrays("mixture10k", 2500, 200, d=64, M=16, ef_construction=48)
    g = [U.build_graph(base, m, 16, 48, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    idx = U.Index(base, g[0], g[1], traverse_dtype="f16")
    q, pd = torch.from_numpy(qs).cuda(), torch.from_numpy(p).cuda()
    bits = int(np.ceil(np.log2(2 * (200 + 32))))
    for nq in (1, 200):
        ref = idx.search(q[:nq], pd[:nq], k=10, ef=200, query_threads=32)
        got = idx.search(q[:nq], pd[:nq], k=10, ef=200, hash_bits=bits, stats=True)
        torch.cuda.synchronize()
        assert torch.equal(ref[0], got[0]) and torch.equal(ref[1], got[1])
        assert (got[2][:, 4] > 0).all()
    assert idx.device_status() == 0
    idx.close()
