"""Mixed path, systems of 40 and more unknowns: the z = 1 samples' two smallest
eigenvalues are down to 1e-14 of the largest apart (noise-free float32 frames,
smooth kernels), where only a double-precision tridiagonal solve finds the null
vector before its one refinement step.  Kernels against the oracle at the mixed
path's bar, 1e-3."""
import numpy as np
import pytest
import torch

import oracle
from cbp_synth.generators import blob_latent, mixture_kernel
from tests._inputs import rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t1,t2", [(20, 20), (25, 15)])
@pytest.mark.parametrize("seed", range(8))
def test_wide_systems_noise_free(gpu_ctx, t1, t2, seed):
    from paper_1203_4874_gb300 import cbp
    rng = np.random.Generator(np.random.PCG64(5000 + 100 * t1 + 10 * t2 + seed))
    lat = blob_latent(rng, 96, 110)
    k1, k2 = mixture_kernel(rng, t1), mixture_kernel(rng, t2)
    b1, b2 = (b.astype(np.float32) for b in oracle.blur_pair(lat, k1, k2))
    prm = cbp.params(t1, t2, path="mixed", flags=cbp.CBP_FLAG_KERNELS_F64)
    g1, g2, _, _ = cbp.cbp_estimate_kernels(gpu_ctx, torch.from_numpy(b1).cuda(), torch.from_numpy(b2).cuda(), prm)
    torch.cuda.synchronize()
    o = oracle.estimate_kernels(b1.astype(np.float64), b2.astype(np.float64), t1, t2)
    assert rel(g1[0].cpu().numpy(), o["k1"]) <= 1e-3 and rel(g2[0].cpu().numpy(), o["k2"]) <= 1e-3
