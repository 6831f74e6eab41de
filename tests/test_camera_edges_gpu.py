"""The camera side where its kernels change their arrangement: the blur's tiles
(16 or 4 rows a thread by the number of blocks) at frame sizes around their
edges, the kernel draws from one entry to the largest, and the coprimality
decisions with the single-precision certificate deciding all, some and none of
the samples.  Blur within the float bound of the forward model (2e-6), kernels
and decisions identical to the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from oracle import camera
from tests._inputs import rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,c,h,w,t", [(1, 1, 1, 1, 1), (1, 2, 30, 31, 2), (1, 1, 31, 33, 3), (2, 1, 112, 48, 17),
                                       (1, 1, 113, 49, 16), (1, 3, 129, 70, 9), (1, 1, 40, 200, 18),
                                       (310, 1, 12, 23, 5), (152, 2, 115, 30, 15), (160, 2, 100, 66, 17)])
def test_blur_tiles(gpu_ctx, n, c, h, w, t):
    from paper_1203_4874_gb300 import cbp
    rng = np.random.default_rng(h * 1000 + w)
    lat = torch.from_numpy(rng.uniform(size=(n, c, h, w)).astype(np.float32))
    k = rng.uniform(size=(n, t, t))
    k /= k.sum(axis=(1, 2), keepdims=True)
    out = cbp.cbp_forward_blur(gpu_ctx, lat.cuda(), torch.from_numpy(k).cuda()).cpu().numpy()
    for f in {0, n // 2, n - 1}:
        for ch in range(c):
            assert rel(out[f, ch], oracle.blur_full(lat[f, ch].double().numpy(), k[f])) <= 2e-6


@pytest.mark.parametrize("t1,t2", [(1, 1), (1, 4), (2, 3), (17, 15), (32, 32)])
@pytest.mark.parametrize("tol", [0.0, 2e-5, 1e-3])
def test_draws_and_decisions(gpu_ctx, t1, t2, tol):
    from paper_1203_4874_gb300 import cbp
    n = 3
    lat = torch.zeros((n, 1, 8, 8), dtype=torch.float64, device="cuda")
    out = cbp.cbp_encrypt(gpu_ctx, lat, t1, t2, seed=31 * t1 + t2, frame0=2, tol=tol, max_attempts=3)
    for f in range(n):
        k1, k2, a = camera.draw_pair(31 * t1 + t2, 2 + f, t1, t2, max(t1, t2), max_attempts=3, tol=tol or 1e-7)
        assert out["attempts"][f] == a
        assert np.array_equal(out["k1"][f].cpu().numpy(), k1) and np.array_equal(out["k2"][f].cpu().numpy(), k2)
