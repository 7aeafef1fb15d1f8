"""Periodic frames far from the origin, bin for bin against the FP64 oracle: their span
decides whether particles are brought home to one cell, and float32 sees it only to
within the rounding of the coordinates.  Integer counts: no tolerance.
"""
import numpy as np
import pytest

import paper_1808_01478_gb300 as dh
import workloads as w

pytestmark = pytest.mark.gpu

BOXES = {"ortho": (w.BOX_ORTHO, w.ortho_box(1.0, 1.1, 1.2)),
         "triclinic": (w.BOX_TRICLINIC, w.triclinic_box(1.0, 1.1, 1.2, *w.C3_ANGLES))}


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("reach", [0.9, 1.5])
@pytest.mark.parametrize("kind", list(BOXES))
@pytest.mark.parametrize("cells", [1e3, 1e5, 1e6, 8388608.25, 1e9])
@pytest.mark.parametrize("span", [0.5, 1.2, 1.98, 3.0])
def test_frames_far_from_the_origin(oracle_mod, span, cells, kind, reach, dtype):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    box_type, box = BOXES[kind]
    s = w.rng_for(26).random((300, 3)) * np.array([span, 0.4, 0.4]) + cells
    s[0] = cells + 0.26  # float32 has one cell's spacing from 2^23 cells on: these two, 1.98 cells
    s[1] = s[0] + np.array([0.99 * span, 0.0, 0.0])  # apart, can round to neighbours
    x = np.ascontiguousarray((s @ w.box_matrix(box).T).astype(dtype))
    offs, nbins = np.array([0, 120, 300]), 200
    r_max = reach * float(w.box_heights(box).min()) / 2.0
    want = oracle_mod.histogram(x, offs, box_type, box, r_max, nbins)
    dev = torch.from_numpy(x).cuda()
    outs = {}
    with dh.Context(0, pool_bytes=64 << 20) as ctx:
        outs["plain"] = ctx.histogram(dev, offs, box_type, box, r_max, nbins)
        fas = [dh.FrameArgs(dev, offs, box_type, box, r_max, nbins) for _ in range(4)]
        ctx.histogram_batch(fas[:2])
        outs["batch"] = fas[1].out
        if dtype == np.float32:
            assert ctx.wait(ctx.submit(fas[2])) == dh.DH_OK
            outs["served"] = fas[2].out
            dh.dh_histogram_noalloc(fas[3].frame)
            outs["noalloc"] = fas[3].out
    for name, out in outs.items():
        got = out.cpu().numpy().view(np.uint64)
        assert np.array_equal(got, want), (name, int(want.sum()), int(got.sum()))
