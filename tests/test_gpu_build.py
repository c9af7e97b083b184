"""The octree at the edges of the build: leaf sizes from 1 to the whole disk, tiles and blocks that end between
moonlets, coincident moonlets down to the deepest level, clusters of every scale.  Cells (level, place, first
moonlet, count, children) equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2310_20374_gb300 import diskgen

pytestmark = pytest.mark.gpu


def scene(n, kind):
    if kind == "disk":
        return diskgen.make_disk(n, 7 + n)["pos"]
    rng = np.random.default_rng(n)
    pos = rng.uniform(-4.0, 4.0, (n, 3))
    if kind == "coincident":                      # groups of nine at one place
        return pos[(np.arange(n) // 9) * 9 % n].copy()
    return pos * 10.0 ** rng.uniform(-7.0, 0.0, (n, 1))   # clusters of every scale around the centre


@pytest.mark.parametrize("kind", ["disk", "coincident", "scales"])
@pytest.mark.parametrize("n,s", [(1, 1), (2, 1), (255, 1), (256, 2), (257, 64), (1000, 999), (1000, 1000), (1000, 1),
                                 (5003, 300), (70001, 64)])
def test_cells_equal_the_oracle(n, s, kind):
    import torch
    from paper_2310_20374_gb300 import ncorp
    pos = np.ascontiguousarray(scene(n, kind))
    m = np.full(n, 1.0 / n)
    cfg = ncorp.ncorp_config_default()
    cfg.precision, cfg.leaf_size = ncorp.NCORP_FP64, s
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        acc = np.zeros((n, 3))
        ncorp.ncorp_accel(ctx, pos, m, n, 1, 0.5, acc)
        cap = 24 * n + 64
        cells, order = np.zeros((cap, 7), dtype=np.int64), np.zeros(n, dtype=np.int64)
        nc = ncorp.ncorp_tree_export(ctx, order=order, cells=cells, cap=cap)
        st = ncorp.ncorp_stats(ctx)
    finally:
        ncorp.ncorp_free(ctx)
    o = oracle.tree_export(oracle.params(p=1, theta=0.5, leaf_size=s), pos, m)
    assert np.array_equal(order, o["order"])
    assert np.array_equal(cells[:nc], o["cells"])
    assert st["leaves"] == int(np.sum(o["cells"][:, 6] == 0)) and st["depth"] == int(o["cells"][:, 0].max())
