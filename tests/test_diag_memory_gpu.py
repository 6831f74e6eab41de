"""Chunked calls bring the diagnostics back into pageable and into pinned memory:
the same values, device-resident and with host I/O."""
import ctypes

import pytest
import torch

from paper_1203_4874_gb300 import cbp

pytestmark = pytest.mark.gpu
FIELDS = ("kappa_max", "gap_min", "sigma_min_max", "scale_resid", "support_ratio", "status", "pad_h", "pad_w")


@pytest.mark.parametrize("host_io", [False, True])
@pytest.mark.parametrize("n", [16, 41])
def test_diagnostics_in_pageable_and_pinned_memory(gpu_ctx, n, host_io):
    g = torch.Generator().manual_seed(n)
    t1, t2 = 5, 4
    b1 = torch.rand((n, 1, 40 + t1 - 1, 52 + t1 - 1), generator=g)
    b2 = torch.rand((n, 1, 40 + t2 - 1, 52 + t2 - 1), generator=g)
    b1, b2 = (b1.pin_memory(), b2.pin_memory()) if host_io else (b1.cuda(), b2.cuda())
    new = (lambda *s: torch.empty(s).pin_memory()) if host_io else (lambda *s: torch.empty(s, device="cuda"))
    prm = cbp.params(t1, t2, path="mixed", flags=cbp.CBP_FLAG_HOST_IO if host_io else 0)
    size = ctypes.sizeof(cbp.cbp_diag) * n
    got = []
    for buf in (torch.zeros(size, dtype=torch.uint8), torch.zeros(size, dtype=torch.uint8).pin_memory()):
        lat, k1, k2 = new(n, 1, 40, 52), new(n, t1, t1), new(n, t2, t2)
        d = (cbp.cbp_diag * n).from_address(buf.data_ptr())
        s = cbp.lib().cbp_deblur_pair(gpu_ctx, ctypes.byref(cbp.frames(b1)), ctypes.byref(cbp.frames(b2)),
                                      ctypes.byref(prm), k1.data_ptr(), k2.data_ptr(), lat.data_ptr(), d,
                                      cbp._stream_ptr(None))
        assert s >= 0
        torch.cuda.synchronize()
        got.append([[getattr(d[i], f) for f in FIELDS] for i in range(n)])
        assert all(row[-1] > 0 for row in got[-1])
    assert got[0] == got[1]
