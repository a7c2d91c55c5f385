"""The GPU builder where its batches hold one node each (the first 32 nodes): it
is then the sequential insertion, and on integer data, whose L1 and L2 sums are
exact, its graph must be the oracle's, row for row as sets.  Caps and beams at
the edges: fewer links than a warp's team, the largest M (rows of 128 links,
more than the 64 slots of one selection pass), efConstruction 1 and past n."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [2, 3, 32, 64])
@pytest.mark.parametrize("efc", [1, 8, 300])
def test_one_node_batches_equal_the_oracle(M, efc):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    for d, metric in ((5, 1), (33, 2), (130, 1)):
        rng = np.random.default_rng(M * 1000 + efc + d)
        base = rng.integers(0, 40, (33, d)).astype(np.float32)
        levels = np.minimum(rng.geometric(0.5, 33) - 1, 4).astype(np.int32)
        got = U.build_graph(base, metric, M, efc, levels, device="gpu")
        ref = oracle.hnsw_build(base, metric, M, efc, levels)
        assert got["num_levels"] == ref["num_levels"] and got["entry_point"] == ref["entry_point"]
        for g, r in zip(got["levels"], ref["levels"]):
            np.testing.assert_array_equal(g["nodes"], r["nodes"])
            for i in range(len(g["nodes"])):
                a = set(g["nbrs"][g["offsets"][i]:g["offsets"][i + 1]].tolist())
                b = set(r["nbrs"][r["offsets"][i]:r["offsets"][i + 1]].tolist())
                assert a == b, (d, metric, i)
