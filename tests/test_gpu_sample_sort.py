"""The sample sort at its edges: one bucket and many, few and many keys in a bucket, equal keys, sorted input, and
keys that differ only between the samples (the radix sort takes over).  Keys are the oracle's and their order is
the stable one; larger sets through the tree's export, on both sides of the most keys it takes."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def sample_places(n):
    b = min(1024, max(1, n // 256, min(256, n // 64)))
    stride = ((n // 4) << 12) // (2 * b)
    j = np.arange(2 * b)
    return (4 * ((j * stride) >> 12)[:, None] + np.arange(4)).ravel()


def scene(n, kind):
    rng = np.random.default_rng(n)
    pos = rng.uniform(-1.0, 1.0, (n, 3))
    if kind == "equal":
        pos[:] = pos[0]
    elif kind == "few":                            # a handful of places (in a large set: of moonlets at a place)
        pos = pos[rng.integers(0, min(n, max(5, n // 40)) if n > 100000 else min(n, 5), n)]
    elif kind == "sorted":
        pos = pos[np.argsort(oracle.keys(pos)[2], kind="stable")]
    elif kind == "between":                        # the samples spread out, all other keys in one octant's corner
        keep = pos[sample_places(n)]
        pos = 0.5 + 1e-3 * pos
        pos[sample_places(n)] = keep
    return np.ascontiguousarray(pos)


@pytest.mark.parametrize("kind", ["uniform", "equal", "few", "sorted", "between"])
@pytest.mark.parametrize("n", [1, 2, 127, 128, 191, 4000, 16384, 20011, 65536])
def test_static_sort(n, kind):
    import torch
    from paper_2310_20374_gb300 import ncorp
    if kind == "between" and n < 4000:
        pytest.skip("every key is a sample or one bucket takes all")
    pos = scene(n, kind)
    dev = torch.tensor(pos, device="cuda")
    keys = torch.empty(n, device="cuda", dtype=torch.int64)
    order = torch.empty(n, device="cuda", dtype=torch.int64)
    for _ in range(2):
        ncorp.ncorp_hilbert_sort_static(dev, n, keys, order, torch.cuda.current_stream().cuda_stream)
        want = np.asarray(oracle.keys(pos)[2]).astype(np.uint64)
        o = np.argsort(want, kind="stable")
        assert np.array_equal(keys.cpu().numpy().astype(np.uint64), want[o])
        assert np.array_equal(order.cpu().numpy(), o)


@pytest.mark.parametrize("n", [200003, (1 << 19) - 1, 1 << 19, (1 << 19) + 1])
@pytest.mark.parametrize("kind", ["uniform", "few", "between"])
def test_tree_order(n, kind):
    import torch
    from paper_2310_20374_gb300 import ncorp
    pos = scene(n, kind if n <= 1 << 19 or kind != "between" else "uniform")
    cfg = ncorp.ncorp_config_default()
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        order = np.zeros(n, dtype=np.int64)
        ncorp.ncorp_accel(ctx, pos, np.full(n, 1.0 / n), n, 1, 0.5, np.zeros((n, 3)))
        ncorp.ncorp_tree_export(ctx, order=order)
    finally:
        ncorp.ncorp_free(ctx)
    want = np.asarray(oracle.keys(pos)[2]).astype(np.uint64)
    assert np.array_equal(order, np.argsort(want, kind="stable"))
