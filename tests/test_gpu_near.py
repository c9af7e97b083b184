"""Near field alone: with thresholds above every product of moonlet counts the walk sums every pair directly, so
the accelerations are the direct sum.  The leaf sizes put the items' target counts at the edges of the kernel's
groups and subsets (one target, odd counts, 32 and 33, 52 and 53, 64 and 65, several subsets of 64)."""
import numpy as np
import pytest

from paper_2310_20374_gb300 import diskgen

pytestmark = pytest.mark.gpu


def direct(pos, m):
    d = pos[None, :, :] - pos[:, None, :]
    r2 = np.einsum("ijk,ijk->ij", d, d)
    with np.errstate(divide="ignore"):
        w = np.where(r2 > 0.0, m[None, :] / (r2 * np.sqrt(r2)), 0.0)
    return np.einsum("ij,ijk->ik", w, d), np.einsum("ij,ij->i", w, np.sqrt(r2))


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n,leaf", [(1, 64), (2, 1), (33, 64), (53, 64), (65, 65), (300, 1), (700, 7), (700, 32), (700, 33),
                                    (700, 52), (700, 53), (700, 64), (701, 130), (1300, 1300)])
def test_direct_sum(n, leaf, fp64):
    import torch
    from paper_2310_20374_gb300 import ncorp
    d = diskgen.make_disk(n, 90 + leaf)
    pos, m = d["pos"].copy(), d["mass"]
    if n > 60:
        pos[n // 2] = pos[3]                      # a coincident pair
        pos[n // 3] = pos[5] + 1e-7               # and a close one
    cfg = ncorp.ncorp_config_default()
    cfg.precision = ncorp.NCORP_FP64 if fp64 else ncorp.NCORP_MIXED
    cfg.leaf_size = leaf
    cfg.n_cs = cfg.n_cc_pre = cfg.n_cc_post = 1 << 30
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        acc, mut = np.zeros((n, 3)), np.zeros((n, 3))
        ncorp.ncorp_accel(ctx, pos, m, n, 3, 0.5, acc, mut)
        assert ncorp.ncorp_stats(ctx)["m2l"] == 0
    finally:
        ncorp.ncorp_free(ctx)
    ref, scale = direct(pos, m)
    # mixed: a term's rounding is a few 2^-24 of it (separation, r^2, the power -3/2 triples it) plus 2^-24 of
    # each of up to 32 partial sums: 40 * 2^-24 of the sum of magnitudes; FP64: the same with 2^-53 and n terms.
    # The close pair's separation in FP32 pairs (48 bits of a position of size 10) carries 2^-48 * 10 / 1e-7.
    tol = 40 * 2.0 ** -24 + 3 * 2.0 ** -48 * 16 / 1e-7 if not fp64 else (n + 40) * 2.0 ** -53
    err = np.linalg.norm(mut - ref, axis=1)
    assert np.all(err <= tol * scale), float(np.max(err / np.maximum(scale, 1e-300)))


@pytest.mark.parametrize("n,leaf", [(1500, 3), (1500, 40), (1500, 64), (1500, 260), (4003, 17), (4003, 700)])
def test_fp64_pairs_serve_both_moonlets(n, leaf):
    """Several leaves and several items a leaf: every pair pulls on both moonlets once (the sum of forces is zero)."""
    import torch
    from paper_2310_20374_gb300 import ncorp
    d = diskgen.make_disk(n, 17 + leaf)
    pos, m = d["pos"].copy(), d["mass"]
    cfg = ncorp.ncorp_config_default()
    cfg.precision, cfg.leaf_size = ncorp.NCORP_FP64, leaf
    cfg.n_cs = cfg.n_cc_pre = cfg.n_cc_post = 1 << 30
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        acc, mut = np.zeros((n, 3)), np.zeros((n, 3))
        ncorp.ncorp_accel(ctx, pos, m, n, 3, 0.5, acc, mut)
    finally:
        ncorp.ncorp_free(ctx)
    ref, scale = direct(pos, m)
    assert np.all(np.linalg.norm(mut - ref, axis=1) <= (n + 40) * 2.0 ** -53 * scale)
    assert np.all(np.abs((m[:, None] * mut).sum(0)) <= (n + 40) * 2.0 ** -53 * (m * scale).sum())
