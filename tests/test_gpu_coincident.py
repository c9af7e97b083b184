"""Coincident moonlets: one place, one acceleration, bit for bit, whatever the order in which the near field's sums are
added; those that share a velocity stay together through a run."""
import numpy as np
import pytest

from paper_2310_20374_gb300 import diskgen

pytestmark = pytest.mark.gpu


def copies(n, of, seed):
    """n moonlets in groups of three at one place, `of` apart in the caller's order"""
    d = diskgen.make_disk(n, seed)
    src = np.arange(n) - of * (np.arange(n) // of % 3)
    d = {k: np.ascontiguousarray(d[k][src] if k in ("pos", "vel") else d[k]) for k in d}
    return d, np.array([np.flatnonzero(src == s)[0] for s in src])   # and the first moonlet at each one's place


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n,leaf,of", [(64, 64, 1), (3000, 40, 7), (4000, 64, 1000), (4001, 200, 1), (2000, 1, 3)])
def test_one_result(n, leaf, of, fp64):
    import torch
    from paper_2310_20374_gb300 import ncorp
    d, root = copies(n, of, 5 + n)
    cfg = ncorp.ncorp_config_default()
    cfg.precision = ncorp.NCORP_FP64 if fp64 else ncorp.NCORP_MIXED
    cfg.leaf_size, cfg.collisions = leaf, 0
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        acc, mut = np.zeros((n, 3)), np.zeros((n, 3))
        ncorp.ncorp_accel(ctx, d["pos"], d["mass"], n, 4, 0.5, acc, mut)
        assert (root != np.arange(n)).sum() >= n // 3
        assert np.array_equal(acc, acc[root]) and np.array_equal(mut, mut[root])
        x, v, m, R = (torch.tensor(d[k], device="cuda") for k in ("pos", "vel", "mass", "radius"))
        for _ in range(40):
            ncorp.ncorp_step(ctx, x, v, m, R, n, 4, 0.5, 1e-2)
        x, v = x.cpu().numpy(), v.cpu().numpy()
        assert np.array_equal(x, x[root]) and np.array_equal(v, v[root])
    finally:
        ncorp.ncorp_free(ctx)


def test_disks_of_a_forest_stay_separate():
    """Two equal disks side by side: their moonlets coincide in pairs, but each disk has its own field."""
    import torch
    from paper_2310_20374_gb300 import ncorp
    n = 500
    d = diskgen.make_disk(n, 8)
    pos = np.concatenate([d["pos"], d["pos"]])
    m = np.concatenate([d["mass"], 3.0 * d["mass"]])
    cfg = ncorp.ncorp_config_default()
    cfg.precision = ncorp.NCORP_FP64
    ctx = ncorp.ncorp_init(cfg, 2 * n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        ncorp.ncorp_set_disks(ctx, [n, n])
        acc, mut = np.zeros((2 * n, 3)), np.zeros((2 * n, 3))
        ncorp.ncorp_accel(ctx, pos, m, 2 * n, 4, 0.5, acc, mut)
    finally:
        ncorp.ncorp_free(ctx)
    assert np.abs(mut[n:] - 3.0 * mut[:n]).max() <= 1e-12 * np.abs(mut).max()
