"""Captured batches are kept for the whole engine, not per stream: more request
shapes than streams, sent again and again from several threads, give the
synchronous call's result bit for bit whichever stream replays them."""
from __future__ import annotations

import threading

import pytest
import torch

from tests.test_serving_gpu import _outputs, _pair, _prm, _wait

pytestmark = pytest.mark.gpu

# ten frame sizes: ten buckets over eight streams
SIZES = [(48 + 4 * i, 64 + 6 * i) for i in range(10)]


@pytest.mark.parametrize("threads", [1, 3])
def test_more_shapes_than_streams(threads):
    from paper_1203_4874_gb300 import cbp
    ctx = cbp.cbp_create(0, 0)
    pairs = [_pair("video_480p", i, h, w) for i, (h, w) in enumerate(SIZES)]
    want = []
    for b1, b2, cfg in pairs:
        lat, k1, k2, _, st = cbp.cbp_deblur_pair(ctx, b1, b2, _prm(cbp, cfg))
        torch.cuda.synchronize()
        assert st >= 0
        want.append((k1, k2, lat))
    bad = []

    def client(first):
        tickets = []
        for k in range(3 * len(pairs)):
            i = (first + k * (1 + first)) % len(pairs)
            b1, b2, cfg = pairs[i]
            prm = _prm(cbp, cfg)
            out = _outputs(cbp, b1, cfg, prm)
            tickets.append((i, cbp.cbp_stream_submit(ctx, b1, b2, prm, *out), out))
        for i, t, out in tickets:
            _wait(cbp, ctx, t)
            if not all(torch.equal(x, y) for x, y in zip(out, want[i])):
                bad.append((first, i))

    ts = [threading.Thread(target=client, args=(f,)) for f in range(threads)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    cbp.cbp_destroy(ctx)
    assert not bad
