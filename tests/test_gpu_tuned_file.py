"""uhnsw_autotune_load takes every configuration that uhnsw_autotune_save can write:
each team width of the warp kernel (4 lanes for rows of up to 12 chunks too) and the
block-per-query kernel; a line that no tuner writes is left out."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_saved_configurations_load(tmp_path):
    import paper_2605_02030_gb300 as pkg
    pkg.build()
    from paper_2605_02030_gb300 import uhnsw as U
    n, d = 50, 96
    base = np.random.default_rng(0).standard_normal((n, d)).astype(np.float32)
    level = {"nodes": np.arange(n, dtype=np.int32), "offsets": np.arange(n + 1, dtype=np.int64),
             "nbrs": np.arange(1, n + 1, dtype=np.int32) % n}
    idx = U.Index(base, {"num_levels": 1, "entry_point": 0, "max_degree0": 1, "max_degree": 1, "n": n,
                         "levels": [level]}, None, traverse_dtype="f16")
    good = [f"1 {d} {64 << i} 16 32 {team} 1536 0 2" for i, team in enumerate((4, 8, 16, 32))]
    good.append(f"1 {d} 64 32 128 0 0 13 0")
    bad = [f"1 {d} 128 32 32 5 1536 0 2", f"1 {d} 256 32 64 8 1536 0 2", f"0 {d} 512 32 32 8 1536 0 2"]
    src, dst = tmp_path / "a.txt", tmp_path / "b.txt"
    src.write_text("\n".join(good + bad) + "\n")
    idx.autotune_load(str(src))
    idx.autotune_save(str(dst))
    assert sorted(dst.read_text().split("\n")) == sorted(good + [""])
    idx.close()
