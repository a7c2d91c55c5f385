"""A stored choice of the warp kernel (uhnsw_autotune, uhnsw_autotune_load) and calls
of few queries: they run as on an index without one, the many as chosen.  The
counters tell the kernels apart: how many L_p terms are summed follows from the
interval of the drop tests (every 1 group in the choice loaded here, every 4 in the
form for few queries), and the ids and distances are the same either way."""
import numpy as np
import pytest

from helpers import workload_arrays
from paper_2605_02030_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("team", [8, 16, 32])
def test_few_queries_ignore_a_stored_warp_kernel(tmp_path, team):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    # integer rows: base sums are exact whatever lanes add them
    w, base, qs, p, _, _ = workload_arrays("sift1m", 3000, 400, d=128, M=16, ef_construction=40)
    g = [U.build_graph(base, m, 16, 40, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    plain, idx = (U.Index(base, g[0], g[1], traverse_dtype="f16") for _ in range(2))
    path = tmp_path / "tuned.txt"
    path.write_text(f"1 128 128 16 32 {team} {4 * 128 * 4} 11 1\n")
    idx.autotune_load(str(path))
    q, pd = torch.from_numpy(qs).cuda(), torch.from_numpy(p).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    row = torch.arange(20 * sms, device="cuda") % len(qs)
    qm, pm = q[row].contiguous(), pd[row].contiguous()
    chosen = dict(query_threads=32, team_lanes=team, stage_bytes=4 * 128 * 4, hash_bits=11, verify_groups=1)
    for persistent in (False, True):
        o = dict(k=10, ef=100, stats=True, persistent=persistent)
        for nq in (1, 7, sms):
            want = plain.search(q[:nq], pd[:nq], **o)
            got = idx.search(q[:nq], pd[:nq], **o)
            warp = plain.search(q[:nq], pd[:nq], **o, **chosen)
            assert all(torch.equal(a, b) for a, b in zip(want, got)), nq
            assert torch.equal(warp[0], got[0]) and torch.equal(warp[1], got[1]), nq
        assert not torch.equal(warp[2][:, 2], got[2][:, 2])
        want = plain.search(qm, pm, **o, **chosen)
        got = idx.search(qm, pm, **o)
        assert all(torch.equal(a, b) for a, b in zip(want, got))
    for x in (plain, idx):
        assert x.device_status() == 0
        x.close()
