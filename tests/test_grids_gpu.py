"""Deconvolution with given kernels over transform grids of every kind: the
smallest, odd and even lengths, lengths with each radix, half-length and
full-length row transforms, one and several columns per strip, kernels from
1 x 1 to 32 x 32.  Against the oracle on its own grid of the same size: FP64
frames within 1e-11 (a transform's rounding, ~1e-15 log2 N, over a denominator
of at least eps = 1e-3 against its largest value of 2); float32 frames on the
mixed path within 1e-4 for the same reason."""
import numpy as np
import pytest
import torch

import oracle
from tests._inputs import rel

pytestmark = pytest.mark.gpu

# (n, c, h, w, t1, t2): latent h x w
GRIDS = [(1, 1, 1, 1, 1, 1), (2, 1, 5, 3, 2, 3), (1, 3, 17, 40, 4, 3), (3, 1, 26, 61, 10, 11), (1, 1, 97, 33, 4, 5),
         (2, 3, 64, 64, 5, 5), (1, 2, 49, 350, 2, 1), (1, 1, 226, 113, 32, 31), (5, 1, 120, 211, 11, 9),
         (1, 1, 480, 640, 17, 15), (1, 3, 719, 1277, 13, 11)]


@pytest.mark.parametrize("n,c,h,w,t1,t2", GRIDS)
@pytest.mark.parametrize("dt,path,bar", [(torch.float64, "fp64", 1e-11), (torch.float32, "mixed", 1e-4)])
def test_given_kernels(gpu_ctx, n, c, h, w, t1, t2, dt, path, bar):
    from paper_1203_4874_gb300 import cbp
    rng = np.random.default_rng(n + 10 * h + 1000 * w)
    eps = 1e-3
    lat = rng.uniform(0.0, 1.0, (n, c, h, w))
    k1, k2 = rng.uniform(0.0, 1.0, (n, t1, t1)), rng.uniform(0.0, 1.0, (n, t2, t2))
    k1 /= k1.sum((1, 2), keepdims=True)
    k2 /= k2.sum((1, 2), keepdims=True)
    b = [oracle.blur_pair(lat[i], k1[i], k2[i]) for i in range(n)]
    np_dt = np.float64 if dt == torch.float64 else np.float32
    b1, b2 = (np.stack([x[k] for x in b]).astype(np_dt) for k in (0, 1))
    prm = cbp.params(t1, t2, path=path, eps=eps, flags=cbp.CBP_FLAG_KERNELS_IN | cbp.CBP_FLAG_KERNELS_F64)
    out = cbp.cbp_deblur_pair(gpu_ctx, torch.from_numpy(b1).cuda(), torch.from_numpy(b2).cuda(), prm,
                              torch.from_numpy(k1).cuda(), torch.from_numpy(k2).cuda())[0]
    torch.cuda.synchronize()
    for i in range(n):
        want = oracle.deconvolve_dual(b1[i].astype(np.float64), b2[i].astype(np.float64), k1[i], k2[i], h, w, eps)
        assert rel(out[i].cpu().numpy(), want) <= bar


@pytest.mark.parametrize("h,w,c,t1,t2,dt,path", [(50, 61, 1, 6, 5, torch.float32, "mixed"),
                                                 (33, 48, 2, 5, 5, torch.float64, "fp64"),
                                                 (24, 1920, 1, 17, 15, torch.float32, "mixed"),
                                                 (24, 1919, 1, 9, 11, torch.float32, "fp64")])
def test_folds_and_transforms_apart_and_together(gpu_ctx, h, w, c, t1, t2, dt, path):
    """A pair alone has blocks of their own for the folds and the transforms, one of
    a batch that fills the GPU shares them: the same bits."""
    from paper_1203_4874_gb300 import cbp
    n = 30
    g = torch.Generator().manual_seed(h + w)
    b1 = torch.rand((n, c, h + t1 - 1, w + t1 - 1), generator=g, dtype=dt).cuda()
    b2 = torch.rand((n, c, h + t2 - 1, w + t2 - 1), generator=g, dtype=dt).cuda()
    for n_ in (8, 15, n):                  # 15 pairs: one chunk
        prm = cbp.params(t1, t2, path=path, eps=1e-3, flags=cbp.CBP_FLAG_KERNELS_F64)
        lat, k1, k2, _, _ = cbp.cbp_deblur_pair(gpu_ctx, b1[:n_], b2[:n_], prm)
        for f in (0, n_ // 2, n_ - 1):
            a = cbp.cbp_deblur_pair(gpu_ctx, b1[f:f + 1], b2[f:f + 1], prm)
            torch.cuda.synchronize()
            assert torch.equal(a[0][0], lat[f]) and torch.equal(a[1][0], k1[f]) and torch.equal(a[2][0], k2[f])
