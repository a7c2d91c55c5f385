"""The server's accounting of search state: a request counts what the kernel that
needs most holds for it.  The block-per-query kernel keeps at least its beam (8 bytes
an entry), the visited table and four buffers of 64 candidates of 8 bytes; with the
kernel left open a request counts no less than with either kernel named."""
import numpy as np
import pytest

from helpers import workload_arrays
from paper_2605_02030_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype,M,ef", [(16, "f32", 8, 16), (128, "f16", 16, 64), (96, "f16", 16, 512)])
def test_state_of_one_request(d, dtype, M, ef):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    w, base, qs, p, _, _ = workload_arrays("mixture10k", 800, 4, d=d, M=M, ef_construction=30)
    g = [U.build_graph(base, m, M, 30, I.graph_levels(w, m), device="gpu") for m in (1, 2)]
    idx = U.Index(base, g[0], g[1], traverse_dtype=dtype)
    state = {}
    for threads in (0, 32, 128):
        srv = U.Server(idx, max_batch=1, streams=1, k_max=10, ef_max=ef, query_threads=threads)
        srv.replay(qs[:1], p[:1], 10, ef, np.zeros(1))
        state[threads] = srv.stats()["peak_state"]
        srv.close()
    table = 4 << max(9, int(np.ceil(np.log2(4 * (ef + 2 * M)))))
    assert state[128] >= 8 * ef + table + 4 * 64 * 8 + 4 * d
    assert state[0] >= max(state[32], state[128] - 4 * 32 * 4)   # (the two may pad a row differently)
    idx.close()
