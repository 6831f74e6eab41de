"""Weight gradients of large batches, where a CTA sums many steps of positions.

Against the oracle's backward pass through the GPU's own activations, at a batch
whose first two layers take four and more steps a CTA (every buffer is refilled):
the bound of test_cnn_gpu.py, seven BF16 roundings.

Against the sum of the pairs' own gradients (a step or two a CTA each): a chunk
is at most 1024 positions, 64 accumulations of 16 products, each truncated by less
than 2^-24 of the sum: 64 2^-24; then the chunks' partials (304, or 512
positions and more each) in eight runs of at most count / 8 and the runs' sums, rounded to nearest, sqrt(count / 8 + 8) 2^-24."""
import math

import numpy as np
import pytest
import torch

from oracle import cnn_oracle as cn
from tests.test_cnn_gpu import _flat, _unflat

pytestmark = pytest.mark.gpu


def frames(n, h, w, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    b1 = torch.rand((n, 1, h, w), device="cuda", generator=g)
    b2 = torch.rand((n, 1, h + 3, w + 3), device="cuda", generator=g)
    kt = torch.rand((n, 2, 15, 15), device="cuda", generator=g)
    return b1, b2, kt / kt.sum(dim=(2, 3), keepdim=True), g


def step(ctx, b1, b2, kt, w):
    from paper_1203_4874_gb300 import cbp
    p, m, v = w.clone(), torch.zeros_like(w), torch.zeros_like(w)
    tr = cbp.cnn_trace_buffers(b1.shape[0], b1.device, grad=True)
    cbp.cbp_cnn_train_step(ctx, b1, b2, kt, p, m, v, step=1, lr=0.0, weight_decay=0.0, trace=tr)
    torch.cuda.synchronize()
    return tr


def test_gradient_against_oracle(gpu_ctx):
    n = 16
    b1, b2, kt, _ = frames(n, 270, 300, 3)
    params = cn.init_params(13)
    w = torch.tensor(_flat(params), dtype=torch.float32, device="cuda")
    tr = step(gpu_ctx, b1, b2, kt, w)
    P = _unflat(w.cpu().numpy())
    ref = None
    for f in range(n):
        z = tr["logits"][f].double().cpu().numpy()
        acts = [tr["input"][f].double().cpu().numpy()] + [a[f].double().cpu().numpy() for a in tr["act"]] + [z]
        K = np.stack([cn.softmax(z[c].ravel()).reshape(15, 15) for c in range(2)])
        g = cn.backward(P, (acts, acts[1:], K), kt[f].double().cpu().numpy())
        ref = [[x / n for x in l] for l in g] if ref is None else [[a + x / n for a, x in zip(r, l)] for r, l in zip(ref, g)]
    got = _unflat(tr["grad"].cpu().numpy())
    for li in range(4):
        for j in range(2):
            # the head's bias gradient is zero in exact arithmetic: against its weights'
            scale = max(np.linalg.norm(ref[li][j]), 1e-3 * np.linalg.norm(ref[li][0]))
            assert np.linalg.norm(got[li][j] - ref[li][j]) < 7 * 2.0 ** -9 * scale, (li, j)


@pytest.mark.parametrize("n", [32, 128, 512])
def test_error_does_not_grow_with_the_batch(gpu_ctx, n):
    b1, b2, kt, g = frames(n, 157, 200, 40 + n)
    w = 0.15 * torch.randn(_flat(cn.init_params(1)).size, device="cuda", generator=g)
    whole = step(gpu_ctx, b1, b2, kt, w)["grad"].double()
    mean = sum(step(gpu_ctx, b1[f:f + 1], b2[f:f + 1], kt[f:f + 1], w)["grad"].double() for f in range(n)) / n
    o = 0
    for side, (c_in, c_out, k, *_) in zip((128, 64, 16), cn.LAYERS):
        nw, count = c_out * c_in * k * k, max(304, n * side * side // 512)
        bound = (64 + math.sqrt(count / 8 + 8)) * 2.0 ** -24
        assert float((whole[o:o + nw] - mean[o:o + nw]).norm() / mean[o:o + nw].norm()) <= bound
        o += nw + c_out
