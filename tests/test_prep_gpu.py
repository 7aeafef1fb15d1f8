"""Preparation of small frames in one launch, against the FP64 oracle bin for bin.

The frames sit on the edges of the launch: one particle, one thread's, one
block's and one cluster's worth and one more (the general path), species of few
particles and empty ones, coordinates of several cells brought home in
double-floats or in binary64 (from 4,096 cells on), both input types and strides,
outputs that are cleared and outputs that are added to.
"""
import numpy as np
import pytest

import paper_1808_01478_gb300 as dh
import workloads as w

pytestmark = pytest.mark.gpu

BOXES = {
    "none": (w.BOX_NONE, np.zeros(9)),
    "ortho": (w.BOX_ORTHO, w.ortho_box(11.0, 12.0, 13.0)),
    "triclinic": (w.BOX_TRICLINIC, w.triclinic_box(12.0, 12.0, 12.0, *w.C3_ANGLES)),
}


@pytest.fixture(scope="module")
def torch_mod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("box", list(BOXES))
@pytest.mark.parametrize("n,cells,dtype,stride", [
    (1, 0, "f4", 3), (2, 0, "f4", 4), (129, 3, "f4", 3), (1024, 0, "f8", 3), (1025, 6000, "f4", 3), (4097, 40, "f4", 4),
    (8192, 2, "f8", 4), (8193, 2000, "f4", 3), (32768, 0, "f4", 3), (32769, 5, "f4", 3)])
def test_small_frames_match_oracle(torch_mod, oracle_mod, box, n, cells, dtype, stride):
    box_type, B = BOXES[box]
    rng = w.rng_for(5000 + n)
    x = rng.random((n, 3))
    if box_type == w.BOX_NONE:
        x = x * 12.0 + 5.0
    else:
        m = w.box_matrix(B)
        x = (x + (rng.integers(-cells, cells + 1, size=(n, 3)) if cells else 0)) @ m.T
    xs = np.zeros((n, stride), dtype)
    xs[:, :3] = x
    cuts = sorted(min(n, k) for k in (1, 1, 130))  # one particle, none, fewer than a run or two, the rest
    offs = np.array([0, *cuts, n], dtype=np.int64)
    r_max, nbins = 5.0, 777
    want = oracle_mod.histogram(np.ascontiguousarray(xs[:, :3]), offs, box_type, B, r_max, nbins)
    with dh.Context(0) as ctx:
        dev = torch_mod.from_numpy(xs).cuda()
        out = torch_mod.full(want.shape, 7, dtype=torch_mod.int64, device="cuda")
        ctx.histogram(dev, offs, box_type, B, r_max, nbins, out)
        assert np.array_equal(out.cpu().numpy().view(np.uint64), want)
        ctx.histogram(dev, offs, box_type, B, r_max, nbins, out, accumulate=True)
        assert np.array_equal(out.cpu().numpy().view(np.uint64), 2 * want)
        assert np.array_equal(ctx.histogram(xs, offs, box_type, B, r_max, nbins), want)


def test_many_species(torch_mod, oracle_mod):
    # a counter group per species, more of them than one thread's share of particles
    n = 300
    x = w.rng_for(77).random((n, 3)).astype(np.float32) * 9.0
    offs = np.arange(n + 1, dtype=np.int64)
    want = oracle_mod.histogram(x, offs, w.BOX_NONE, np.zeros(9), 8.0, 3)
    with dh.Context(0) as ctx:
        got = ctx.histogram(torch_mod.from_numpy(x).cuda(), offs, w.BOX_NONE, None, 8.0, 3)
    assert np.array_equal(got.cpu().numpy().view(np.uint64), want)


@pytest.mark.parametrize("box", list(BOXES))
@pytest.mark.parametrize("n,nbins", [(1, 5), (2, 5), (129, 60000), (8193, 9000), (32769, 700), (65536, 700),
                                     (65536, 20000), (65537, 700)])
def test_allocation_free_frames_match_dh_histogram(torch_mod, box, n, nbins):
    # both ways through the fixed scratch: ordered for the list kernel where everything
    # fits (not with 65,536 particles and 20,000 bins, nor with 65,537), and in place
    box_type, B = BOXES[box]
    m = np.eye(3) * 12.0 if box_type == w.BOX_NONE else w.box_matrix(B)
    x = torch_mod.from_numpy((w.rng_for(6000 + n).random((n, 3)) @ m.T).astype(np.float32)).cuda()
    offs = np.array([0, n // 3, n // 3, n], dtype=np.int64)
    with dh.Context(0) as ctx:
        want = ctx.histogram(x, offs, box_type, B, 5.0, nbins)
    out = torch_mod.full((6, nbins), 7, dtype=torch_mod.int64, device="cuda")
    dh.dh_histogram_noalloc(dh.FrameArgs(x, offs, box_type, B, 5.0, nbins, out).frame)
    assert torch_mod.equal(out, want)
    dh.dh_histogram_noalloc(dh.FrameArgs(x, offs, box_type, B, 5.0, nbins, out, True).frame)
    assert torch_mod.equal(out, 2 * want)


@pytest.mark.parametrize("n,cuts,box,shape", [
    (15999, [], "ortho", "uniform"),               # one particle short of the strips: the curve
    (16000, [], "ortho", "uniform"),
    (16000, [2047, 4095], "triclinic", "uniform"),  # one species in the curve's order, two in strips
    (20001, [1, 1, 3000], "ortho", "flat"),        # a plane: every particle in one cell of an axis
    (32768, [16384], "triclinic", "point"),        # half of them in one place
    (33025, [129], "ortho", "long"),               # general path, sides 1 : 1 : 60
    (33025, [], "triclinic", "cells"),             # ... brought home from several cells
    (200000, [], "none", "uniform"),
])
def test_strip_order(torch_mod, oracle_mod, n, cuts, box, shape):
    box_type, B = BOXES[box]
    if shape == "long":
        B = w.ortho_box(6.0, 6.0, 360.0)
    rng = w.rng_for(7000 + n)
    x = rng.random((n, 3))
    if shape == "flat":
        x[:, 1] = 0.25
    if shape == "point":
        x[: n // 2] = 0.5 + 1e-4 * x[: n // 2]
    if shape == "cells":
        x += rng.integers(-3, 4, size=(n, 3))
    m = np.eye(3) * 12.0 if box_type == w.BOX_NONE else w.box_matrix(B)
    x = (x @ m.T).astype(np.float32)
    offs = np.array([0, *cuts, n], dtype=np.int64)
    r_max, nbins = (2.9 if shape == "long" else 5.0), 600
    want = oracle_mod.histogram(x, offs, box_type, B, r_max, nbins)
    with dh.Context(0) as ctx:
        got = ctx.histogram(torch_mod.from_numpy(x).cuda(), offs, box_type, B, r_max, nbins)
    assert np.array_equal(got.cpu().numpy().view(np.uint64), want)


@pytest.mark.parametrize("box", list(BOXES))
def test_served_request_without_room_for_the_order(torch_mod, box):
    # 36 bytes a particle are enough for a request to be taken, 60 for its ordered copies
    box_type, B = BOXES[box]
    n, nbins = 45_000, 600
    x = torch_mod.from_numpy((w.rng_for(91).random((n, 3)) * 10.0).astype(np.float32)).cuda()
    offs = np.array([0, n // 2, n], dtype=np.int64)
    with dh.Context(0, pool_bytes=2 << 20, max_inflight=2) as c:
        want = c.histogram(x, offs, box_type, B, 5.0, nbins)
        fa = dh.FrameArgs(x, offs, box_type, B, 5.0, nbins)
        assert c.wait(c.submit(fa)) == dh.DH_OK
        assert torch_mod.equal(fa.out, want)
        big = torch_mod.zeros((60_000, 3), device="cuda")
        with pytest.raises(dh.DHError) as e:
            c.submit(dh.FrameArgs(big, [0, 60_000], box_type, B, 5.0, nbins))
        assert e.value.status == dh.DH_ERR_NOMEM


@pytest.mark.parametrize("species,nbins", [(1, 16384), (1, 16385), (3, 16384), (16, 2000)])
@pytest.mark.parametrize("n", [90, 1100])
def test_outputs_cleared_by_the_preparation_or_by_a_fill(torch_mod, oracle_mod, n, species, nbins):
    # 16,384 words per block of the launch (one block for 90 particles, two for 1,100) and one more
    x = (w.rng_for(92).random((n, 3)) * 8.0).astype(np.float32)
    offs = np.array([n * k // species for k in range(species + 1)], dtype=np.int64)
    want = oracle_mod.histogram(x, offs, w.BOX_NONE, np.zeros(9), 14.0, nbins)
    dev = torch_mod.from_numpy(x).cuda()
    with dh.Context(0, pool_bytes=256 << 20) as ctx:
        for accumulate in (False, True):
            fas = [dh.FrameArgs(dev, offs, w.BOX_NONE, None, 14.0, nbins,
                                torch_mod.full(want.shape, 3, dtype=torch_mod.int64, device="cuda"), accumulate)
                   for _ in range(5)]
            ctx.histogram(dev, offs, w.BOX_NONE, None, 14.0, nbins, fas[0].out, accumulate=accumulate)
            ctx.histogram_batch(fas[1:3])
            assert ctx.wait(ctx.submit(fas[3])) == dh.DH_OK
            dh.dh_histogram_noalloc(fas[4].frame)
            for k, fa in enumerate(fas):
                assert np.array_equal(fa.out.cpu().numpy().view(np.uint64), want + (3 if accumulate else 0)), (k, accumulate)
        assert np.array_equal(ctx.histogram(x, offs, w.BOX_NONE, None, 14.0, nbins), want)  # host arrays
