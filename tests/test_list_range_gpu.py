"""Frames on the edge of what the list kernel's float32 positions can hold, bin for
bin against the FP64 oracle: particles so far away that their squared distance in
bins passes the float32 range, and bins so narrow that every distance does.  Integer
counts: no tolerance.
"""
import numpy as np
import pytest

import paper_1808_01478_gb300 as dh
import workloads as w

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_mod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def check(torch, oracle_mod, x, offs, box_type, box, r_max, nbins):
    """Plain, batched, served and allocation-free calls (float32 for the last two)."""
    x = np.ascontiguousarray(x)
    offs = np.asarray(offs, np.int64)
    want = oracle_mod.histogram(x, offs, box_type, box, r_max, nbins)
    dev = torch.from_numpy(x).cuda()
    got = {}
    with dh.Context(0, pool_bytes=64 << 20) as ctx:
        got["plain"] = ctx.histogram(dev, offs, box_type, box, r_max, nbins)
        fas = [dh.FrameArgs(dev, offs, box_type, box, r_max, nbins) for _ in range(4)]
        ctx.histogram_batch(fas[:2])
        got["batch"] = fas[1].out
        if x.dtype == np.float32:
            assert ctx.wait(ctx.submit(fas[2])) == dh.DH_OK
            got["served"] = fas[2].out
            dh.dh_histogram_noalloc(fas[3].frame)
            got["noalloc"] = fas[3].out
    for name, out in got.items():
        assert np.array_equal(out.cpu().numpy().view(np.uint64), want), (name, int(want.sum()), int(out.sum()))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("at", [1e10, 1e13, 1e18, 1e20, 1e30, 3e38])
@pytest.mark.parametrize("sizes", [[100], [700], [90, 300]], ids=lambda s: "-".join(map(str, s)))
def test_particles_parked_far_away(torch_mod, oracle_mod, sizes, at, dtype):
    offs = np.concatenate([[0], np.cumsum(sizes)])
    n = int(offs[-1])
    x = (w.rng_for(21).random((n, 3)) * 10.0).astype(np.float32).astype(dtype)
    x[n // 2] = (at, 1.0, 2.0)
    x[n - 1] = (at, 1.0, 2.0)  # two in one place
    x[1] = (3.0, -at, -at)
    check(torch_mod, oracle_mod, x, offs, w.BOX_NONE, np.zeros(9), 17.0, 1000)


@pytest.mark.parametrize("kind", ["none", "ortho", "triclinic"])
@pytest.mark.parametrize("r_max", [1e-9, 1e-17, 1e-36, 1e-42])
def test_bins_far_narrower_than_the_frame(torch_mod, oracle_mod, kind, r_max):
    # only particles in one place, and some next to each other, are inside r_max
    box_type, box = {"none": (w.BOX_NONE, np.zeros(9)), "ortho": (w.BOX_ORTHO, w.ortho_box(9.0, 8.0, 10.0)),
                     "triclinic": (w.BOX_TRICLINIC, w.triclinic_box(9, 8, 10, *w.C3_ANGLES))}[kind]
    x = (w.rng_for(22).random((400, 3)) * 7.0).astype(np.float32)
    x[200:] = x[:200]
    x[0] = 0.0
    x[1:40] = (w.rng_for(23).random((39, 3)) * min(2.0 * r_max, 1e-9)).astype(np.float32)
    check(torch_mod, oracle_mod, x, [0, 150, 400], box_type, box, r_max, 100)


def test_a_box_far_longer_than_wide(torch_mod, oracle_mod):
    box = w.ortho_box(1e25, 10.0, 11.0)
    x = (w.rng_for(24).random((500, 3)) * 10.0).astype(np.float32)
    x[:, 0] = w.rng_for(25).choice(np.array([0.0, 1e24, 5e24, 9e24]), 500)
    check(torch_mod, oracle_mod, x, [0, 200, 500], w.BOX_ORTHO, box, 5.0, 300)
