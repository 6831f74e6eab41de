"""Mixed path around the sizes at which the scale solve's float-float stage stops
fitting in a CTA's shared memory: its layout falls just under the device's limit
there, but not beside the kernel's own static arrays.  Kernels against the
oracle at the mixed path's bar, 1e-3."""
import numpy as np
import pytest
import torch

import oracle
from tests._inputs import rel
from tests.test_team_solver_gpu import make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t1,t2,m", [(28, 13, 0), (28, 14, 0), (28, 15, 0), (28, 16, 0), (27, 19, 0),
                                     (13, 13, 29), (13, 14, 29), (6, 5, 30), (6, 6, 30), (7, 6, 30)])
def test_scale_stage_at_the_shared_memory_limit(gpu_ctx, t1, t2, m):
    from paper_1203_4874_gb300 import cbp
    b1, b2 = make_pair(100 * t1 + t2, 72, 81, t1, t2)
    prm = cbp.params(t1, t2, m=m, path="mixed", flags=cbp.CBP_FLAG_KERNELS_F64)
    k1, k2, _, _ = cbp.cbp_estimate_kernels(gpu_ctx, torch.from_numpy(b1).cuda(), torch.from_numpy(b2).cuda(), prm)
    torch.cuda.synchronize()
    o = oracle.estimate_kernels(b1.astype(np.float64), b2.astype(np.float64), t1, t2, m or None)
    assert rel(k1[0].cpu().numpy(), o["k1"]) <= 1e-3 and rel(k2[0].cpu().numpy(), o["k2"]) <= 1e-3
