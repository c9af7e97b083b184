"""Near field of a small cluster far from the origin, in units in which the distance squared leaves the FP32 range: the
sums are those of the separations, whatever the number of sources that pads the last chunk."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 30, 31, 63, 66, 130])
def test_far_from_the_origin(n, fp64):
    import torch
    from paper_2310_20374_gb300 import ncorp
    rng = np.random.default_rng(n)
    pos = 1e20 + rng.uniform(-1e12, 1e12, (n, 3))
    m = rng.uniform(0.5, 1.5, n) * 1e6
    cfg = ncorp.ncorp_config_default()
    cfg.precision = ncorp.NCORP_FP64 if fp64 else ncorp.NCORP_MIXED
    cfg.leaf_size = 256
    cfg.n_cs = cfg.n_cc_pre = cfg.n_cc_post = 1 << 30
    ctx = ncorp.ncorp_init(cfg, n, 0, torch.cuda.current_stream().cuda_stream)
    try:
        acc, mut = np.zeros((n, 3)), np.zeros((n, 3))
        ncorp.ncorp_accel(ctx, pos, m, n, 3, 0.5, acc, mut)
    finally:
        ncorp.ncorp_free(ctx)
    d = pos[None, :, :] - pos[:, None, :]
    r = np.linalg.norm(d, axis=2)
    w = np.where(r > 0.0, m[None, :] / np.where(r > 0.0, r, 1.0) ** 3, 0.0)
    ref, scale = np.einsum("ij,ijk->ik", w, d), (w * r).sum(1)
    # as for a disk near the origin (40 roundings of a term), and mixed: the FP32 pairs carry 2^-48 of 1e20 a
    # component, 3 components of 2 moonlets, tripled by the power -3/2, against the least separation
    close = 3 * 6 * 2.0 ** -48 * 1e20 / r[r > 0].min()
    tol = (n + 40) * 2.0 ** -53 if fp64 else 40 * 2.0 ** -24 + close
    err = np.linalg.norm(mut - ref, axis=1)
    assert np.all(err <= tol * scale), float(np.max(err / scale))
