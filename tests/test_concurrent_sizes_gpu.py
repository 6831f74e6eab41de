"""Calls of different sizes at the same time, each thread with a context and a
stream of its own, beside a serving engine that captures new request shapes:
the kernels' shared-memory limits are state of the process, and no caller's size
may become another's limit.  Every call succeeds and gives what it gives alone,
bit for bit."""
import threading

import pytest
import torch

from tests.test_serving_gpu import _outputs, _pair, _prm

pytestmark = pytest.mark.gpu

# t1, t2, height, width, path: shared memory from a few KB to the largest
CALLS = [(5, 4, 64, 64, "mixed"), (15, 17, 300, 420, "mixed"), (25, 24, 100, 100, "mixed"), (9, 11, 240, 320, "fp64")]


def test_calls_of_many_sizes_at_once(gpu_ctx):
    from paper_1203_4874_gb300 import cbp
    bad = []

    def frames(t1, t2, h, w):
        g = torch.Generator(device="cuda").manual_seed(100 * t1 + t2)
        return (torch.rand((1, 1, h + t - 1, w + t - 1), device="cuda", generator=g) for t in (t1, t2))

    def caller(t1, t2, h, w, path):
        ctx, st = cbp.cbp_create(0), torch.cuda.Stream()
        try:
            with torch.cuda.stream(st):
                b1, b2 = frames(t1, t2, h, w)
                prm = cbp.params(t1, t2, path=path, eps=1e-4)
                outs = [cbp.cbp_deblur_pair(ctx, b1, b2, prm)[:3] for _ in range(300)]
                st.synchronize()
                want = alone[t1, t2]
                bad.extend(("result", t1, t2) for o in outs if not all(torch.equal(x, y) for x, y in zip(o, want)))
        except cbp.CbpError as e:
            bad.append((str(e), t1, t2))
        finally:
            st.synchronize()
            cbp.cbp_destroy(ctx)

    def server():
        ctx, tickets = cbp.cbp_create(0), []
        for i in range(24):        # a new shape each: a capture each
            b1, b2, cfg = _pair("video_480p", 0, 48 + 8 * i, 64 + 9 * i)
            prm = _prm(cbp, cfg, "mixed")
            out = _outputs(cbp, b1, cfg, prm)
            tickets.append((cbp.cbp_stream_submit(ctx, b1, b2, prm, *out), b1, b2, out))
        for i, (t, *_) in enumerate(tickets):
            status, _ = cbp.cbp_stream_poll(ctx, t, -1)
            if status < 0:
                bad.append((cbp.status_string(status), "serving", i))
        cbp.cbp_destroy(ctx)

    alone = {}
    for t1, t2, h, w, path in CALLS:
        b1, b2 = frames(t1, t2, h, w)
        alone[t1, t2] = cbp.cbp_deblur_pair(gpu_ctx, b1, b2, cbp.params(t1, t2, path=path, eps=1e-4))[:3]
    torch.cuda.synchronize()
    threads = [threading.Thread(target=caller, args=a) for a in CALLS] + [threading.Thread(target=server)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad[:5]
