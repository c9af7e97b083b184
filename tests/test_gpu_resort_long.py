"""The nearly-sorted key sort where a thread holds more keys than it remembers as movers (over 64: above 2.5e6 keys on
152 SMs): those past the 64th are looked at a second time."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt,path", [(1e-7, 1), (1e-4, 2)])
def test_long_runs(dt, path):
    import torch
    from paper_2310_20374_gb300 import ncorp
    n = 64 * 256 * torch.cuda.get_device_properties(0).multi_processor_count + 120011
    rng = np.random.default_rng(3)
    r, phi = rng.uniform(2.0, 10.0, n), rng.uniform(0.0, 2.0 * np.pi, n)
    pos = np.stack([r * np.cos(phi), r * np.sin(phi), 0.01 * rng.normal(size=n)], axis=1)
    vel = np.stack([-np.sin(phi), np.cos(phi), np.zeros(n)], axis=1) / np.sqrt(r)[:, None]
    cfg = ncorp.ncorp_config_default()
    cfg.collisions = 0
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        x, v = torch.tensor(pos, device="cuda"), torch.tensor(vel, device="cuda")
        m, R = torch.full((n,), 1e-12, device="cuda", dtype=torch.float64), torch.full((n,), 1e-6, device="cuda",
                                                                                     dtype=torch.float64)
        for _ in range(2):
            ncorp.ncorp_step(ctx, x, v, m, R, n, 1, 0.7, dt)
        order, keys = np.zeros(n, dtype=np.int64), np.zeros(n, dtype=np.uint64)
        ncorp.ncorp_tree_export(ctx, order=order, keys=keys)
        assert ncorp.ncorp_stats(ctx)["sort_path"] == path
    finally:
        ncorp.ncorp_free(ctx)
    want = np.asarray(oracle.keys(x.cpu().numpy())[2]).astype(np.uint64)
    o = np.argsort(want, kind="stable")
    assert np.array_equal(order, o) and np.array_equal(keys, want[o])
