"""The climbs' FP32-guided maxima and opening angles against the oracle bit for bit where the estimates are of
little use: leaves of one moonlet, moonlets equidistant from their centre, clusters far from the origin and much
smaller than their distance, large and small units, zero radii and velocities, extreme mass ratios."""
import numpy as np
import pytest

import oracle
from paper_2310_20374_gb300 import diskgen

pytestmark = pytest.mark.gpu


def scene(kind, n):
    d = diskgen.make_disk(n, 31)
    pos, vel, m, R = d["pos"].copy(), d["vel"].copy(), d["mass"].copy(), d["radius"].copy()
    if kind == "lattice":
        k = int(round(n ** (1 / 3))) + 1
        pos = np.stack(np.meshgrid(*[np.arange(k) * 0.25] * 3, indexing="ij"), -1).reshape(-1, 3)[:n].astype(float)
        m, vel, R = np.full(n, 1.0 / n), np.full((n, 3), 0.125), np.full(n, 0.0625)
    elif kind == "tight":     # groups of 20 within 1e-9 of points of size 10
        rng = np.random.default_rng(4)
        pos = pos[(np.arange(n) // 20) * 20 % n] + 1e-9 * rng.standard_normal((n, 3))
    elif kind == "large":
        pos, vel, R, m = pos * 1e30, vel * 1e25, R * 1e25, m * 1e25
    elif kind == "small":
        pos, vel, R, m = pos * 1e-25, vel * 1e-25, R * 1e-25, m * 1e-25
    elif kind == "still":
        vel, R = np.zeros_like(vel), np.zeros_like(R)
    elif kind == "masses":
        m = 10.0 ** np.random.default_rng(5).uniform(-14.0, 0.0, n)
    return [np.ascontiguousarray(a) for a in (pos, vel, m, R)]


@pytest.mark.parametrize("theta", [0.02, 0.5, 0.95])
@pytest.mark.parametrize("s", [1, 16])
@pytest.mark.parametrize("kind", ["lattice", "tight", "large", "small", "still", "masses"])
def test_geometry_bit_exact(kind, s, theta):
    import torch
    from paper_2310_20374_gb300 import ncorp
    n, dt = 1500, 1e-3
    pos, vel, m, R = scene(kind, n)
    cfg = ncorp.ncorp_config_default()
    cfg.precision, cfg.leaf_size = ncorp.NCORP_FP64, s
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    cap = 24 * n
    gg, cg = np.zeros((cap, 6)), np.zeros((cap, 5))
    try:
        acc = np.zeros((n, 3))
        ncorp.ncorp_accel(ctx, pos, m, n, 1, theta, acc)
        nc = ncorp.ncorp_tree_export(ctx, ggeo=gg, cap=cap)
        ncorp.ncorp_collide(ctx, pos, vel, R, n, dt)
        assert ncorp.ncorp_tree_export(ctx, cgeo=cg, cap=cap) == nc
    finally:
        ncorp.ncorp_free(ctx)
    o = oracle.tree_export(oracle.params(p=1, theta=theta, leaf_size=s), pos, m, vel, R, dt)
    assert np.array_equal(gg[:nc], o["ggeo"])
    assert np.array_equal(cg[:nc], o["cgeo"])
