"""Shared-memory counts of the list kernel where the shortest of several images is
chosen pair by pair: a block's 32-bit words must reach the 64-bit histogram before
they pass 2^31, whichever way the pairs were counted.
"""
import numpy as np
import pytest

import paper_1808_01478_gb300 as dh
import workloads as w

pytestmark = pytest.mark.gpu


def test_chosen_images_are_flushed_too(tmp_path):
    # a slab so thin that every pair has several images to choose from, and one bin
    # that takes every pair: each of the blocks counts about 3.3e9 of them
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 1_000_000
    box = np.array([10.0, 1000.0, 1000.0])
    x = torch.from_numpy((w.rng_for(31).random((n, 3)) * box).astype(np.float32)).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert n * (n - 1) // 2 // sms > 2 ** 31
    path = tmp_path / "tune.txt"  # the list kernel, by the last column
    path.write_text("".join(f"{sms} 1 {wl} 20 0 1024 256 1 1 1.0 0 1\n" for wl in range(3)))
    with dh.Context(0, tune_cache=str(path)) as ctx:
        out = ctx.histogram(x, [0, n], w.BOX_ORTHO, w.ortho_box(*box), 710.0, 1)
        st = ctx.stats()
    assert st["blocks"] <= sms and st["block_threads"] == 512, st
    assert int(out.cpu().numpy().view(np.uint64)[0, 0]) == n * (n - 1) // 2
