"""Device memory the serving engine holds, as the allocator counts it (the
process's default pool, which nothing else here allocates from)."""
import ctypes
import os
import subprocess
import sys
from pathlib import Path

import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = Path(__file__).resolve().parents[1]

RESERVED_NOW, RESERVED_HIGH, USED_NOW = 5, 6, 7      # cudaMemPoolAttrReservedMemCurrent, -High, UsedMemCurrent


class Pool:
    """The default memory pool of device 0."""

    def __init__(self):
        self.rt = ctypes.CDLL("libcudart.so.13")
        self.h = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.h), 0) == 0

    def used(self, attr=USED_NOW):
        v = ctypes.c_uint64()
        assert self.rt.cudaMemPoolGetAttribute(self.h, attr, ctypes.byref(v)) == 0
        return v.value

    def reset_high(self):
        assert self.rt.cudaMemPoolSetAttribute(self.h, RESERVED_HIGH, ctypes.byref(ctypes.c_uint64(0))) == 0


@pytest.fixture
def pool(built_lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.synchronize()
    return Pool()


def request(h, w, t1=7, t2=8, c=1):
    from paper_1203_4874_gb300 import cbp
    b1, b2 = (torch.rand((1, c, h + t - 1, w + t - 1), device="cuda") for t in (t1, t2))
    out = (torch.empty((1, t1, t1), device="cuda"), torch.empty((1, t2, t2), device="cuda"),
           torch.empty((1, c, h, w), device="cuda"))
    return b1, b2, cbp.params(t1, t2, path="mixed", eps=1e-4), out


def submit(ctx, r):
    from paper_1203_4874_gb300 import cbp
    return cbp.cbp_stream_submit(ctx, *r[:3], *r[3])


def wait(ctx, t):
    from paper_1203_4874_gb300 import cbp
    s, _ = cbp.cbp_stream_poll(ctx, t, -1)
    return s


def test_kept_batches_are_bounded(pool):
    """48 request shapes one after the other: 32 workspaces stay."""
    from paper_1203_4874_gb300 import cbp
    ctx = cbp.cbp_create(0)
    before, one = pool.used(), 0
    for i in range(48):
        assert wait(ctx, submit(ctx, request(120 + 2 * i, 160))) >= 0
        one = max(one, cbp.cbp_workspace_size(*request(120 + 2 * i, 160)[:3]) + (1 << 12))
    held = pool.used() - before
    cbp.cbp_destroy(ctx)
    assert held <= 32 * one
    torch.cuda.synchronize()
    assert pool.used() == before


def test_room_for_a_new_shape_while_another_batch_runs(pool):
    """A kept batch gives its workspace to a new shape while the stream it was
    captured on runs something else: the pool takes no more memory from the device."""
    from paper_1203_4874_gb300 import cbp
    kept, long, new = request(720, 1280), request(480, 640, 25, 24), request(700, 1270)
    sizes = [cbp.cbp_workspace_size(*r[:3]) for r in (kept, long, new)]
    assert sizes[2] <= sizes[0]
    for _ in range(3):
        base = pool.used()                       # other contexts' workspaces
        ctx = cbp.cbp_create(0, sizes[0] + sizes[1] + (1 << 16))     # tables and alignment
        for r in (long, kept):                   # both captured on the first stream
            assert wait(ctx, submit(ctx, r)) >= 0
        torch.cuda.synchronize()
        before = pool.used(RESERVED_NOW)
        pool.reset_high()
        tickets = [submit(ctx, long), submit(ctx, new)]
        assert all(wait(ctx, t) >= 0 for t in tickets)
        high = pool.used(RESERVED_HIGH)
        cbp.cbp_destroy(ctx)
        torch.cuda.synchronize()
        assert high <= before
        assert pool.used() == base


# cudaMallocAsync that fails as often as it is told to, then passes through
SHIM = """
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static int left;
void fail_next(int n) { left = n; }
int cudaMallocAsync(void** p, size_t bytes, void* stream) {
  if (left > 0) { --left; return 2; }   /* cudaErrorMemoryAllocation */
  int (*real)(void**, size_t, void*) = 0;
  void* h = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
  *(void**)&real = dlsym(h, "cudaMallocAsync");
  return real(p, bytes, stream);
}
"""
CHILD = """
import ctypes, sys
from tests.test_serving_memory_gpu import request, submit, wait
from paper_1203_4874_gb300 import cbp
shim = ctypes.CDLL(sys.argv[1])
ctx = cbp.cbp_create(0)
for h in (100, 120, 140):
    assert wait(ctx, submit(ctx, request(h, 160))) >= 0
out = []
for fails in (1, 2, 50, 0):
    shim.fail_next(fails)
    out.append(wait(ctx, submit(ctx, request(180 + fails, 160))))
    shim.fail_next(0)
cbp.cbp_destroy(ctx)
print(*out)
"""


def test_device_out_of_memory(built_lib, tmp_path):
    """Allocations that fail within the budget: kept batches are given up until
    one succeeds; with none left the request is refused, and the next one runs."""
    from paper_1203_4874_gb300 import cbp
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, lib = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, str(lib)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, LD_PRELOAD=str(lib)))
    assert r.returncode == 0, r.stderr[-3000:]
    assert [int(x) for x in r.stdout.split()] == [0, 0, cbp.CBP_ERR_BUDGET, 0]
