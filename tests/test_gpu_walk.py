"""The walk where its first block hands over to all of them: trees whose frontiers stay within, just pass and far
exceed what one block keeps, from one moonlet up.  Cell decisions equal the oracle's and FP64 accelerations agree."""
import numpy as np
import pytest

import oracle
from paper_2310_20374_gb300 import diskgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["disk", "ball", "coincident"])
@pytest.mark.parametrize("n,s", [(1, 1), (2, 1), (9, 1), (60, 1), (120, 1), (250, 1), (500, 2), (1000, 17), (2500, 17),
                                 (6001, 40)])
def test_decisions_equal_the_oracle(n, s, kind):
    import torch
    from paper_2310_20374_gb300 import ncorp
    rng = np.random.default_rng(n)
    pos = diskgen.make_disk(n, 3 + n)["pos"] if kind == "disk" else rng.uniform(-2.0, 2.0, (n, 3))
    if kind == "coincident":
        pos = pos[(np.arange(n) // 4) * 4]
    pos, m = np.ascontiguousarray(pos), rng.uniform(0.5, 1.5, n) / n
    th = (4, 0, 0)   # many small interactions: frontiers as large as the tree allows
    cfg = ncorp.ncorp_config_default()
    cfg.precision, cfg.leaf_size = ncorp.NCORP_FP64, s
    cfg.n_cs, cfg.n_cc_pre, cfg.n_cc_post = th
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    acc, mut = np.zeros((n, 3)), np.zeros((n, 3))
    try:
        ncorp.ncorp_accel(ctx, pos, m, n, 3, 0.5, acc, mut)
        st = ncorp.ncorp_stats(ctx)
    finally:
        ncorp.ncorp_free(ctx)
    P = oracle.params(p=3, theta=0.5, leaf_size=s, gravity_thresholds=th)
    want, ost = oracle.falcon_accel(P, pos, m)
    assert [st[k] for k in ("cells", "m2l", "p2p_pairs", "p2p_self", "p2p_interactions")] == \
           [ost[k] for k in ("cells", "m2l", "p2p_pairs", "p2p_self", "p2p_interactions")]
    assert np.abs(mut - want).max() <= 1e-11 * np.abs(want).max()
