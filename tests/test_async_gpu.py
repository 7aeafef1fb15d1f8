"""Asynchronous calls on a busy stream: their descriptors are uploaded from one pinned
buffer, which the next call must not write before the upload has run, and their
workspace must not be used on another stream before they are done.
"""
import numpy as np
import pytest

import paper_1808_01478_gb300 as dh
import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("streams", [1, 2])
def test_calls_behind_other_work(streams):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = w.rng_for(61)
    box = w.ortho_box(14.0)
    frames = [(torch.from_numpy((rng.random((n, 3)) * 14.0).astype(np.float32)).cuda(), [0, n // 3, n], 4.0 + 0.4 * k)
              for k, n in enumerate((3000, 500, 4000, 1200, 2500, 40_000))]
    with dh.Context(0) as ctx:
        want = [ctx.histogram(x, o, w.BOX_ORTHO, box, r, 300) for x, o, r in frames]
        outs = [torch.full((3, 300), 7, dtype=torch.int64, device="cuda") for _ in frames]
        side = [torch.cuda.Stream() for _ in range(streams)]
        torch.cuda.synchronize()
        keep = []
        for k, ((x, o, r), out) in enumerate(zip(frames, outs)):
            stream = side[k % streams]
            with torch.cuda.stream(stream):
                torch.cuda._sleep(20_000_000)  # some 10 ms of other work first
            ctx.set_stream(stream)
            keep.append(ctx.histogram_async(x, o, w.BOX_ORTHO, box, r, 300, out))
        ctx.sync()
        ctx.set_stream(None)
        torch.cuda.synchronize()
    for k, (got, expect) in enumerate(zip(outs, want)):
        assert torch.equal(got, expect), k
