"""Pairs that overlap, touch or nearly touch at the start of the step, at rest or not, on scales from tiny to the
disk's: the pairs found by the tree search are the brute-force oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-3, 1e-9, 1e-14])
@pytest.mark.parametrize("speed", [0.0, 1e-12, 1e-4, 1.0])
def test_pairs_equal_brute_force(scale, speed):
    import torch
    from paper_2310_20374_gb300 import ncorp
    rng = np.random.default_rng(int(-np.log10(scale)) * 7 + int(speed * 3))
    n = 1200
    centre = rng.uniform(-1.0, 1.0, (n // 2, 3))
    rad = scale * rng.uniform(0.3, 1.0, n)
    f = np.tile([0.0, 0.5, 1.0 - 2.0 ** -6, 1.0 - 2.0 ** -8, 1.0 - 2.0 ** -30, 1.0, 1.0 + 2.0 ** -30, 1.0 + 2.0 ** -8, 1.2, 2.0],
                n // 20)
    way = rng.normal(size=(n // 2, 3))
    way /= np.linalg.norm(way, axis=1)[:, None]
    pos = np.empty((n, 3))
    pos[0::2] = centre                                   # partners at f (R1 + R2)
    pos[1::2] = centre + way * (f * (rad[0::2] + rad[1::2]))[:, None]
    vel = np.repeat(rng.normal(size=(n // 2, 3)), 2, axis=0)
    vel[1::2] -= speed * scale * way * rng.choice([-1.0, 0.0, 1.0], n // 2)[:, None]
    vel[1::2] += 0.1 * speed * scale * rng.normal(size=(n // 2, 3))
    dt = 0.7
    cfg = ncorp.ncorp_config_default()
    cfg.leaf_size = 20
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        buf = np.zeros((1 << 16, 2), dtype=np.int64)
        ncorp.ncorp_collide(ctx, np.ascontiguousarray(pos), np.ascontiguousarray(vel), rad, n, dt)
        k = ncorp.ncorp_collisions(ctx, buf, len(buf))
    finally:
        ncorp.ncorp_free(ctx)
    want = oracle.collide_brute(pos, vel, rad, dt)
    want = np.asarray(want[0] if isinstance(want, tuple) else want).reshape(-1, 2)
    assert np.array_equal(buf[:k], want[np.lexsort((want[:, 1], want[:, 0]))])
