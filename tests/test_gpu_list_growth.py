"""Walk lists that fill up in any generation: the call grows them and reruns, it does not fail.

The capacities (NCORP_TEST_LIST_CAP, read by ncorp_init) run from one the head of the walk fills to one that only the
last generations do, so that some of them are first exceeded in the generation the head hands over to all the blocks,
before their first grid barrier."""
import numpy as np
import pytest

from paper_2310_20374_gb300 import diskgen

pytestmark = pytest.mark.gpu

CAPS = [200, 700, 1500, 3000, 6000, 12000, 40000]


def context(cfg, n, monkeypatch, cap=None):
    import torch
    from paper_2310_20374_gb300 import ncorp
    if cap:
        monkeypatch.setenv("NCORP_TEST_LIST_CAP", str(cap))
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    monkeypatch.delenv("NCORP_TEST_LIST_CAP", raising=False)
    return ctx


def accel(monkeypatch, d, cap=None):
    from paper_2310_20374_gb300 import ncorp
    n = len(d["mass"])
    cfg = ncorp.ncorp_config_default()
    cfg.precision, cfg.leaf_size = ncorp.NCORP_FP64, 17
    cfg.n_cs, cfg.n_cc_pre, cfg.n_cc_post = 4, 0, 0   # many cell pairs
    ctx = context(cfg, n, monkeypatch, cap)
    try:
        acc, mut = np.zeros((n, 3)), np.zeros((n, 3))
        ncorp.ncorp_accel(ctx, d["pos"], d["mass"], n, 3, 0.5, acc, mut)
        return mut, ncorp.ncorp_stats(ctx)
    finally:
        ncorp.ncorp_free(ctx)


@pytest.fixture(scope="module")
def disk():
    return diskgen.make_disk(20000, 71)


@pytest.mark.parametrize("cap", CAPS)
def test_gravity_lists(monkeypatch, disk, cap):
    ref, rst = accel(monkeypatch, disk)
    got, st = accel(monkeypatch, disk, cap)
    assert rst["m2l"] > max(CAPS)   # every capacity is exceeded
    assert [st[k] for k in ("cells", "m2l", "p2p_pairs", "p2p_self", "p2p_interactions")] == \
           [rst[k] for k in ("cells", "m2l", "p2p_pairs", "p2p_self", "p2p_interactions")]
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()   # (the order of sums is the lists')


@pytest.mark.parametrize("cap", CAPS[:-1])
def test_collision_lists(monkeypatch, cap):
    from paper_2310_20374_gb300 import ncorp
    n = 20000
    d = diskgen.make_disk(n, 72, a_lo=2.0, a_hi=2.5, r_lo=1e-2, r_hi=2e-2, sigma_e=0.1, sigma_i=0.05)
    got = []
    for c in (None, cap):
        cfg = ncorp.ncorp_config_default()
        cfg.leaf_size = 8
        ctx = context(cfg, n, monkeypatch, c)
        try:
            ncorp.ncorp_collide(ctx, d["pos"], d["vel"], d["radius"], n, 1e-2)
            pairs = np.zeros((1 << 17, 2), dtype=np.int64)
            k = ncorp.ncorp_collisions(ctx, pairs, len(pairs))
            got.append((pairs[:k], ncorp.ncorp_stats(ctx)))
        finally:
            ncorp.ncorp_free(ctx)
    (ref, rst), (pairs, st) = got
    assert rst["col_pairs"] > max(CAPS[:-1])
    assert len(ref) > 0 and np.array_equal(pairs, ref)
    assert st["col_pairs"] == rst["col_pairs"] and st["col_tests"] == rst["col_tests"]


def direct_on_gpu(pos, m):
    import torch
    out = torch.empty_like(pos)
    for i in range(0, len(pos), 2000):
        d = pos[None, :, :] - pos[i:i + 2000, None, :]
        r2 = (d * d).sum(2)
        w = torch.where(r2 > 0, m[None, :] * r2.pow(-1.5), 0.0)
        out[i:i + 2000] = (w[:, :, None] * d).sum(1)
    return out


@pytest.mark.parametrize("fp64", [False, True])
def test_near_items_grow_alone(fp64):
    """Large leaves, every pair summed directly: several near-field items an entry.  One rerun that grows the items to
    what the walk counted, not reruns that double the other lists; the same in a step, for both tree sets."""
    import torch
    from paper_2310_20374_gb300 import ncorp
    n, leaf = 50000, 256
    d = diskgen.make_disk(n, 73)
    pos, vel, m, R = (torch.tensor(d[k], device="cuda") for k in ("pos", "vel", "mass", "radius"))
    cfg = ncorp.ncorp_config_default()
    cfg.precision = ncorp.NCORP_FP64 if fp64 else ncorp.NCORP_MIXED
    cfg.leaf_size, cfg.collisions = leaf, 0
    cfg.n_cs = cfg.n_cc_pre = cfg.n_cc_post = 1 << 30
    ref = direct_on_gpu(pos, m)
    scale = ref.norm(dim=1).max()
    stream = torch.cuda.current_stream().cuda_stream
    ctx = ncorp.ncorp_init(cfg, n, 0, stream)
    try:
        free = torch.cuda.mem_get_info()[0]
        launches = []
        for _ in range(2):
            acc, mut = torch.empty_like(pos), torch.empty_like(pos)
            ncorp.ncorp_accel(ctx, pos, m, n, 3, 0.5, acc, mut)
            launches.append(ncorp.ncorp_stats(ctx)["launches"])
            # FP64: n terms' rounding; mixed: 40 * 2^-24 of the sum of magnitudes (below 1e3 of the result's scale)
            assert float((mut - ref).norm(dim=1).max()) <= ((n + 40) * 2.0 ** -53 if fp64 else 40 * 2.0 ** -24) * 1e3 * scale
        assert launches[0] == 2 * launches[1], launches
        assert free - torch.cuda.mem_get_info()[0] <= 8 << 20   # (the other lists' doubling takes 16 MB and more)
    finally:
        ncorp.ncorp_free(ctx)
    states = []
    for grown in (False, True):   # a step that meets the full list in its own tree, and one that does not
        ctx = ncorp.ncorp_init(cfg, n, 0, stream)
        try:
            if grown:
                ncorp.ncorp_accel(ctx, pos, m, n, 3, 0.5, torch.empty_like(pos), None)
            x, v = pos.clone(), vel.clone()
            for _ in range(3):
                ncorp.ncorp_step(ctx, x, v, m, R, n, 3, 0.5, 1e-3)
            assert ncorp.ncorp_stats(ctx)["graph"] == 1
            states.append((x, v))
        finally:
            ncorp.ncorp_free(ctx)
    tol = 1e-13 if fp64 else 1e-9
    assert float((states[0][0] - states[1][0]).abs().max()) <= tol * float(pos.abs().max())
    assert float((states[0][1] - states[1][1]).abs().max()) <= tol * float(vel.abs().max())
