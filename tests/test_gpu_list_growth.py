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
