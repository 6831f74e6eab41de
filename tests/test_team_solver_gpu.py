"""The per-sample and scale solves where they change their arrangement: system
widths n = t1 + t2 and 2 M on both sides of 32 (one or two matrix columns per
lane) and at the smallest and largest supported, batches of few and of many
samples to an SM.  Kernels against the oracle at the repository's bars: 1e-9
(FP64 path), 1e-3 (mixed path); pairs of a large batch against the same pairs
alone within twice the bar, and the same bits."""
import numpy as np
import pytest
import torch

import oracle
from tests._inputs import rel

pytestmark = pytest.mark.gpu


def make_pair(seed, h, w, t1, t2, c=1, sigma=1e-3):
    rng = np.random.default_rng(seed)
    lat = rng.uniform(0.0, 1.0, (c, h, w))
    k1, k2 = rng.uniform(0.0, 1.0, (t1, t1)), rng.uniform(0.0, 1.0, (t2, t2))
    b1, b2 = oracle.blur_pair(lat, k1 / k1.sum(), k2 / k2.sum())
    b1 = b1 + rng.normal(0.0, sigma, b1.shape)
    b2 = b2 + rng.normal(0.0, sigma, b2.shape)
    return [b.astype(np.float32) for b in (b1, b2)]


@pytest.mark.parametrize("t1,t2,m", [(1, 2, 0), (2, 2, 0), (5, 4, 0), (16, 15, 0), (16, 16, 0), (17, 16, 0),
                                     (3, 2, 16), (3, 2, 17), (24, 20, 0), (32, 32, 0)])
@pytest.mark.parametrize("path,bar", [("fp64", 1e-9), ("mixed", 1e-3)])
def test_system_widths(gpu_ctx, t1, t2, m, path, bar):
    from paper_1203_4874_gb300 import cbp
    b1, b2 = make_pair(100 * t1 + t2, 72, 81, t1, t2)
    prm = cbp.params(t1, t2, m=m, path=path, flags=cbp.CBP_FLAG_KERNELS_F64)
    k1, k2, _, _ = cbp.cbp_estimate_kernels(gpu_ctx, torch.from_numpy(b1).cuda(), torch.from_numpy(b2).cuda(), prm)
    torch.cuda.synchronize()
    o = oracle.estimate_kernels(b1.astype(np.float64), b2.astype(np.float64), t1, t2, m or None)
    assert rel(k1[0].cpu().numpy(), o["k1"]) <= bar and rel(k2[0].cpu().numpy(), o["k2"]) <= bar


@pytest.mark.parametrize("path", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [38, 39])   # 8 samples a pair: 304 and 312
def test_batches_around_a_cta_per_sample(gpu_ctx, n, path):
    from paper_1203_4874_gb300 import cbp
    pairs = [make_pair(7000 + f, 40, 45, 6, 5) for f in range(4)]
    B1, B2 = (torch.from_numpy(np.stack([pairs[f % 4][k] for f in range(n)])).cuda() for k in (0, 1))
    prm = cbp.params(6, 5, path=path, flags=cbp.CBP_FLAG_KERNELS_F64)
    stages = cbp.cbp_estimate_kernels_stages(gpu_ctx, B1, B2, prm)     # one batch, not split
    torch.cuda.synchronize()
    tol = 2e-9 if path == "fp64" else 2e-3
    for f in range(4):
        k1, k2, _, _ = cbp.cbp_estimate_kernels(gpu_ctx, B1[f:f + 1], B2[f:f + 1], prm)
        torch.cuda.synchronize()
        for g in range(f, n, 4):
            assert rel(stages["k1"][g].cpu().numpy(), k1[0].cpu().numpy()) <= tol
            assert rel(stages["k2"][g].cpu().numpy(), k2[0].cpu().numpy()) <= tol


@pytest.mark.parametrize("path", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [7, 40])
def test_a_pair_does_not_depend_on_its_batch(gpu_ctx, n, path):
    """Bit for bit: the serving engine's batches give what each request gives alone."""
    from paper_1203_4874_gb300 import cbp
    pairs = [make_pair(7100 + f, 40, 45, 6, 5, c=3) for f in range(n)]
    B1, B2 = (torch.from_numpy(np.stack([p[k] for p in pairs])).cuda() for k in (0, 1))
    prm = cbp.params(6, 5, path=path, flags=cbp.CBP_FLAG_KERNELS_F64)
    lat, k1, k2, diag, _ = cbp.cbp_deblur_pair(gpu_ctx, B1, B2, prm)     # 40 pairs: two chunks
    torch.cuda.synchronize()
    for f in range(0, n, 3):
        a = cbp.cbp_deblur_pair(gpu_ctx, B1[f:f + 1], B2[f:f + 1], prm)
        torch.cuda.synchronize()
        assert torch.equal(a[0][0], lat[f]) and torch.equal(a[1][0], k1[f]) and torch.equal(a[2][0], k2[f])
        assert all(getattr(a[3][0], x) == getattr(diag[f], x) for x in
                   ("kappa_max", "gap_min", "scale_resid", "support_ratio", "pad_h", "pad_w", "status"))
