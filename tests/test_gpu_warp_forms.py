"""The warp kernel's forms (24 or 32 warps per SM by the launch's shared memory,
two queries per block) against the block-per-query kernel: beams on both sides
of the sizes where 32 warps fit, rows of one to four chunks a lane, odd and
tiny batches, plain and persistent.  The rows hold integers, so that base sums
are exact whatever lanes add them, and the L_p sums are added by the same lanes
in both kernels: ids and distances are equal bit for bit."""
import numpy as np
import pytest

from helpers import workload_arrays
from paper_2605_02030_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype", [(30, "f32"), (60, "f32"), (128, "f32"), (250, "f32"), (500, "f32"),
                                     (96, "f16"), (96, "bf16"), (128, "f16")])
def test_forms_equal_the_block_kernel(d, dtype):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    # L2 sums stay below 2^24 (exact in FP32): values up to 255, 180 for 500 dimensions
    w, base, qs, p, _, _ = workload_arrays("sift1m", 2500, 1301, d=d, M=16, ef_construction=40)
    if d > 250:
        base, qs = np.minimum(base, 180.0), np.minimum(qs, 180.0)
    base, qs = np.ascontiguousarray(base, np.float32), np.ascontiguousarray(qs, np.float32)
    p = p.copy()
    p[::5], p[1::5], p[2::5] = 1.0, 2.0, 0.5
    g = [U.build_graph(base, m, 16, 40, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    idx = U.Index(base, g[0], g[1], traverse_dtype=dtype)
    q, pd = torch.from_numpy(qs).cuda(), torch.from_numpy(p).cuda()
    for nq in (1, 3, 1301):
        for ef in (10, 64, 96, 120, 220, 400):
            for k, width, pers in ((10, 1, False), (ef, 3, True)):
                o = dict(k=k, ef=ef, width=width, persistent=pers)
                ref = idx.search(q[:nq], pd[:nq], query_threads=128, **o)
                got = idx.search(q[:nq], pd[:nq], query_threads=32, **o)
                torch.cuda.synchronize()
                assert torch.equal(ref[0], got[0]) and torch.equal(ref[1], got[1]), (nq, o)
    assert idx.device_status() == 0
    idx.close()
