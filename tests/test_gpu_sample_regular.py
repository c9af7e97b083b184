"""The sample sort on inputs stored regularly (rows, rings): the samples split them as well as unordered ones, so that
the sort takes about as long; and on keys that differ only between its samples, which the radix sort takes over."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def static_sort(pos, repeats=1):
    """keys, order and the least time of a call in us"""
    import torch
    from paper_2310_20374_gb300 import ncorp
    n = len(pos)
    dev = torch.tensor(np.ascontiguousarray(pos), device="cuda")
    keys = torch.empty(n, device="cuda", dtype=torch.int64)
    order = torch.empty(n, device="cuda", dtype=torch.int64)
    stream, best = torch.cuda.current_stream().cuda_stream, float("inf")
    for _ in range(repeats):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        ncorp.ncorp_hilbert_sort_static(dev, n, keys, order, stream)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, 1e3 * e0.elapsed_time(e1))
    return keys.cpu().numpy().astype(np.uint64), order.cpu().numpy(), best


def check(pos, keys, order):
    want = np.asarray(oracle.keys(np.ascontiguousarray(pos))[2]).astype(np.uint64)
    o = np.argsort(want, kind="stable")
    assert np.array_equal(keys, want[o]) and np.array_equal(order, o)


def rows(n, width):
    i = np.arange(n)
    return np.stack([(i // width) / (n // width), (i % width) / width, np.zeros(n)], axis=1)


def rings(n, width):
    i = np.arange(n)
    r, phi = 2.0 + (i // width) / (n // width), 2.0 * np.pi * (i % width) / width
    return np.stack([r * np.cos(phi), r * np.sin(phi), np.zeros(n)], axis=1)


@pytest.mark.parametrize("scene", [rows, rings])
@pytest.mark.parametrize("n,width", [(16384, 32), (16384, 64), (65536, 64), (65536, 128)])
def test_regular_input(n, width, scene):
    plain = np.random.default_rng(1).normal(size=(n, 3))
    least = static_sort(plain, 50)[2]
    pos = scene(n, width)
    keys, order, us = static_sort(pos, 50)
    check(pos, keys, order)
    # a split that fails adds the radix sort's eight passes to the samples': 2.0 to 2.6 times an unordered input's time
    assert us <= 1.7 * least, (us, least)


def sample_places(n):
    b = min(1024, max(1, n // 256, min(256, n // 64)))
    lg = 0 if n > 1 << 18 else 1
    runs = (8 * b) >> lg
    stride = ((n >> lg) << 12) // runs
    r = np.arange(runs, dtype=np.uint64)
    a = (r * np.uint64(stride)) >> np.uint64(12)
    room = (((r + np.uint64(1)) * np.uint64(stride)) >> np.uint64(12)) - a
    mask = np.uint64(0xffffffff)
    h = ((r + np.uint64(1)) * np.uint64(0x9e3779b1)) & mask
    h = ((h ^ (h >> np.uint64(15))) * np.uint64(0x85ebca77)) & mask
    h ^= h >> np.uint64(13)
    first = (a + ((h * room) >> np.uint64(32))) << np.uint64(lg)
    return (first[:, None] + np.arange(1 << lg, dtype=np.uint64)).ravel().astype(np.int64)


@pytest.mark.parametrize("n", [1 << 18, (1 << 18) + 1, 7 << 16, (7 << 16) + 1])
def test_order_beside_the_lines(n):
    """On both sides of the most keys sampled in runs, and of the most the sample sort takes."""
    import torch
    from paper_2310_20374_gb300 import ncorp
    pos = np.random.default_rng(n).uniform(-1.0, 1.0, (n, 3))
    pos[:n // 8] = pos[n // 8:2 * (n // 8)]   # some places twice
    ctx = ncorp.ncorp_init(ncorp.ncorp_config_default(), n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        order = np.zeros(n, dtype=np.int64)
        ncorp.ncorp_accel(ctx, pos, np.full(n, 1.0 / n), n, 1, 0.5, np.zeros((n, 3)))
        ncorp.ncorp_tree_export(ctx, order=order)
    finally:
        ncorp.ncorp_free(ctx)
    want = np.asarray(oracle.keys(pos)[2]).astype(np.uint64)
    assert np.array_equal(order, np.argsort(want, kind="stable"))


@pytest.mark.parametrize("n", [4000, 20011, 65536, 131072, 300001])
def test_keys_between_the_samples(n):
    """All keys but the samples in one octant's corner: more than a bucket holds."""
    import torch
    from paper_2310_20374_gb300 import ncorp
    pos = np.random.default_rng(n).uniform(-1.0, 1.0, (n, 3))
    at = sample_places(n)
    assert len(np.unique(at)) == len(at) and at.max() < n
    keep = pos[at]
    pos = 0.5 + 1e-3 * pos
    pos[at] = keep
    if n <= 65536:
        keys, order, _ = static_sort(pos)
        check(pos, keys, order)
    ctx = ncorp.ncorp_init(ncorp.ncorp_config_default(), n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        order = np.zeros(n, dtype=np.int64)
        ncorp.ncorp_accel(ctx, pos, np.full(n, 1.0 / n), n, 1, 0.5, np.zeros((n, 3)))
        ncorp.ncorp_tree_export(ctx, order=order)
    finally:
        ncorp.ncorp_free(ctx)
    want = np.asarray(oracle.keys(pos)[2]).astype(np.uint64)
    assert np.array_equal(order, np.argsort(want, kind="stable"))
