"""Weight gradients over the chunks of positions: a batch's gradient is the mean
of its pairs' own (each pair's activations do not depend on the batch, and with
a power of two of pairs the scaled gradients round to BF16 alike), whatever the
split of the positions into chunks, which changes with the number of pairs.
FP32 sums of at most 2^12 terms a chunk, then of the chunks: a few times
sqrt(2^12) 2^-24 = 4e-6 of a layer's gradient; bound 1e-4, far below a chunk's
share (1/304)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

LAYERS = ((576, 32), (9216, 32), (9216, 32), (256, 2))


@pytest.mark.parametrize("n", [2, 8, 32])
def test_batch_gradient_is_the_mean(gpu_ctx, n):
    from paper_1203_4874_gb300 import cbp
    g = torch.Generator(device="cuda").manual_seed(40 + n)
    b1 = torch.rand((n, 1, 257, 300), device="cuda", generator=g)
    b2 = torch.rand((n, 1, 260, 303), device="cuda", generator=g)
    w = 0.15 * torch.randn(cbp.cbp_cnn_param_count(), device="cuda", generator=g)
    kt = torch.rand((n, 2, 15, 15), device="cuda", generator=g)
    kt /= kt.sum(dim=(2, 3), keepdim=True)

    def grad(sl):
        p, m, v = w.clone(), torch.zeros_like(w), torch.zeros_like(w)
        tr = {"grad": torch.empty_like(w)}
        cbp.cbp_cnn_train_step(gpu_ctx, b1[sl], b2[sl], kt[sl], p, m, v, step=1, lr=0.0, weight_decay=0.0, trace=tr)
        torch.cuda.synchronize()
        return tr["grad"].double().cpu().numpy()

    whole = grad(slice(0, n))
    mean = sum(grad(slice(f, f + 1)) for f in range(n)) / n
    o = 0
    for nw, nb in LAYERS:
        ref = mean[o:o + nw]
        assert np.linalg.norm(whole[o:o + nw] - ref) <= 1e-4 * np.linalg.norm(ref)
        # the head's bias gradient is zero in exact arithmetic: against its weights'
        scale = max(np.linalg.norm(mean[o + nw:o + nw + nb]), 1e-3 * np.linalg.norm(ref))
        assert np.linalg.norm(whole[o + nw:o + nw + nb] - mean[o + nw:o + nw + nb]) <= 1e-4 * scale
        o += nw + nb
