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


@pytest.mark.parametrize("n,cuts", [(3000, []), (3000, [1000]), (40_000, [20_000]), (210_000, [])])
def test_few_far_particles_leave_the_order_of_the_others(torch_mod, n, cuts):
    # runs stay compact, so hardly more pairs are re-decided than without them: three far
    # particles' runs with every other pair, and 3 times the rest
    x = (w.rng_for(28).random((n, 3)) * 30.0).astype(np.float32)
    far = x.copy()
    far[[5, n // 2, n - 1], [0, 1, 2]] = (1e20, -7e4, 2e6)
    offs = np.array([0, *cuts, n])
    share = {}
    with dh.Context(0) as ctx:
        for name, y in (("near", x), ("far", far)):
            ctx.histogram(torch_mod.from_numpy(y).cuda(), offs, w.BOX_NONE, None, 52.0, 5000)
            st = ctx.stats()
            share[name] = st["deferred"] / st["pairs"]
    assert share["far"] < 3.0 * share["near"] + 3 * 128 / n * 2, share


@pytest.mark.parametrize("nbins", [1, 700, 300_000])
def test_pairs_of_a_far_particle_s_run(torch_mod, oracle_mod, nbins):
    # decided in float32 where that is enough: lattice distances on the bin edges, particles
    # in one place, and pairs beyond r_max among them
    g = np.arange(9, dtype=np.float32) * 0.5
    x = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    x = np.concatenate([x, x[::3], np.array([[1e12, 0, 0], [1e12, 0.5, 0], [0, -2e15, 1e9]], np.float32)])
    x = x[w.rng_for(29).permutation(len(x))]
    check(torch_mod, oracle_mod, x, [0, 300, len(x)], w.BOX_NONE, np.zeros(9), 3.5, min(nbins, 60_000))
    if nbins > 60_000:  # (beyond the allocation-free limit)
        want = oracle_mod.histogram(x, np.array([0, 300, len(x)]), w.BOX_NONE, np.zeros(9), 3.5, nbins)
        with dh.Context(0) as ctx:
            got = ctx.histogram(torch_mod.from_numpy(x).cuda(), [0, 300, len(x)], w.BOX_NONE, None, 3.5, nbins)
        assert np.array_equal(got.cpu().numpy().view(np.uint64), want)
