"""The size scan where its kernels change their arrangement: frame sides around
the blocks of columns (128), rows (4) and loads in flight (16), strided and
double-precision frames, one candidate and the widest range.  Ratios above the
scan's floor against the oracle's within 1e-6 and every one within the floor of
double rounding in the normal matrix (2e-7, ten times 1e-8 and more); sizes and
the excluded candidates identical."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,w,t1,t2,c,dtype,tmin,tmax", [
    (60, 123, 3, 3, 1, torch.float32, 3, 3), (61, 125, 5, 4, 2, torch.float32, 1, 32),
    (124, 128, 4, 5, 1, torch.float64, 2, 12), (33, 47, 2, 7, 3, torch.float32, 1, 32),
    (16, 15, 1, 1, 1, torch.float32, 1, 8)])
def test_scan(gpu_ctx, h, w, t1, t2, c, dtype, tmin, tmax):
    from paper_1203_4874_gb300 import cbp
    rng = np.random.default_rng(h * w)
    pairs = []
    for _ in range(2):
        lat = rng.uniform(0.0, 1.0, (c, h, w))
        k1, k2 = rng.uniform(0.0, 1.0, (t1, t1)), rng.uniform(0.0, 1.0, (t2, t2))
        pairs.append(oracle.blur_pair(lat, k1 / k1.sum(), k2 / k2.sum()))
    b = [torch.from_numpy(np.stack([p[k] for p in pairs])).to(dtype) for k in (0, 1)]
    # rows two elements apart from the next: a strided batch
    wide = [torch.zeros(x.shape[:-1] + (x.shape[-1] + 2,), dtype=dtype, device="cuda") for x in b]
    views = [y[..., :x.shape[-1]].copy_(x) for x, y in zip(b, wide)]
    g1, g2, found, r = cbp.cbp_estimate_size(gpu_ctx, views[0], views[1], tmin, tmax)
    for f in range(2):
        o1, o2, of, ratios = oracle.estimate_size(b[0][f].double().numpy(), b[1][f].double().numpy(), tmin, tmax)
        got = {tmin + i: float(v) for i, v in enumerate(r[f])} if r.shape[1] == tmax - tmin + 1 else \
            {max(tmin, t1 - t2 + 1, 1) + i: float(v) for i, v in enumerate(r[f])}
        for t, v in got.items():
            if v < 0 or t not in ratios:
                continue
            assert abs(v - ratios[t]) <= max(2e-7, 1e-6 * ratios[t])
        if dtype == torch.float64:
            assert (g1[f], g2[f], found[f]) == (o1, o2, of)
