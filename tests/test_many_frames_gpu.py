"""Batches of very many frames: more species than a launch dimension holds, and
frames that need another preparation than the rest.
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


@pytest.mark.parametrize("odd", ["none", "empty", "large", "wide"])
def test_more_species_than_a_launch_dimension(torch_mod, oracle_mod, odd):
    # 66,000 frames of three particles, and one that the one-launch preparation cannot take
    frames, nbins, r_max = 66_000, 2, 2.0
    rng = w.rng_for(41)
    x = torch_mod.from_numpy(rng.random((frames * 3, 3)).astype(np.float32)).cuda()
    out = torch_mod.full((frames, 1, nbins), 9, dtype=torch_mod.int64, device="cuda")
    fas = [dh.FrameArgs(x[3 * k:3 * k + 3], [0, 3], w.BOX_NONE, None, r_max, nbins, out[k]) for k in range(frames)]
    if odd != "none":
        n, bins = {"empty": (0, 3), "large": (40_000, 50), "wide": (2000, 50_000)}[odd]
        y = (rng.random((n, 3)) * 5.0).astype(np.float32)
        want = oracle_mod.histogram(y, np.array([0, n // 3, n]), w.BOX_NONE, np.zeros(9), 4.0, bins)
        fas.insert(frames // 2, dh.FrameArgs(torch_mod.from_numpy(y).cuda(), [0, n // 3, n], w.BOX_NONE, None, 4.0, bins))
    with dh.Context(0) as ctx:
        ctx.histogram_batch(fas)
    got = out.cpu().numpy()
    d = np.linalg.norm(np.diff(np.concatenate([x.cpu().numpy().astype(np.float64).reshape(-1, 3, 3)] * 2, 1)[:, :4], axis=1),
                       axis=2)  # the three distances
    near = (d < r_max / 2).sum(1)
    assert np.array_equal(got[:, 0, 0], near) and np.array_equal(got[:, 0, 1], 3 - near)
    if odd != "none":
        assert np.array_equal(fas[frames // 2].out.cpu().numpy().view(np.uint64), want)


@pytest.mark.parametrize("box", ["none", "ortho"])
def test_segments_of_one_block_and_of_many(torch_mod, oracle_mod, box):
    # 300 frames of three species, each species pair one block's own, and a frame whose
    # species pairs are shared by blocks; the smallest have one particle a species
    rng = w.rng_for(42)
    frames = []
    for k in range(300):
        n = 20_000 if k == 170 else int(rng.integers(3, 700))
        side = (n / 0.1) ** (1.0 / 3.0)
        b = w.ortho_box(side)
        kind, r = (w.BOX_NONE, 2.0 * side) if box == "none" else (w.BOX_ORTHO, 0.5 * side)
        cuts = [0, n // 3, n // 2, n]
        frames.append(w.frame_from((rng.random((n, 3)) * side).astype(np.float32), cuts, kind, b, r, 400, str(k)))
    fas = [dh.FrameArgs(torch_mod.from_numpy(f.coords).cuda(), f.offsets, f.box_type, f.box, f.r_max, f.nbins)
           for f in frames]
    with dh.Context(0) as ctx:
        ctx.histogram_batch(fas)
    for fa, f in zip(fas, frames):
        assert np.array_equal(fa.out.cpu().numpy().view(np.uint64), oracle_mod.histogram_frame(f)), f.name


def test_time_of_a_batch_is_linear_in_its_frames(torch_mod):
    # four times the frames take four times as long (2 at most for the rest), not sixteen
    n, most = 600, 2000
    x = torch_mod.from_numpy((w.rng_for(43).random((most, n, 3)) * 18.0).astype(np.float32)).cuda()
    out = torch_mod.zeros((most, 6, 300), dtype=torch_mod.int64, device="cuda")
    ms = {}
    with dh.Context(0, flags=dh.DH_CFG_TIMING) as ctx:
        for frames in (most // 4, most):
            fas = [dh.FrameArgs(x[k], [0, 200, 400, n], w.BOX_NONE, None, 32.0, 300, out[k]) for k in range(frames)]
            runs = []
            for _ in range(4):
                ctx.histogram_batch(fas)
                runs.append(ctx.stats()["pair_kernel_ms"])
            ms[frames] = min(runs)
    assert int(out.sum()) == most * (n * (n - 1) // 2)
    assert ms[most] < 8.0 * ms[most // 4], ms


@pytest.mark.parametrize("where", ["device", "host"])
def test_empty_frames_leave_the_preparation_of_the_others_alone(torch_mod, oracle_mod, where):
    # the first, one between and the last frame empty: their outputs are cleared (or left, to
    # be added to), the others are prepared in the one launch they take without them
    rng = w.rng_for(44)
    sizes = [0, 700, 0, 1300, 40, 0]
    xs = [(rng.random((n, 3)) * 9.0).astype(np.float32) for n in sizes]
    box = w.ortho_box(9.0)
    offs = [np.array([0, n // 4, n]) for n in sizes]
    want = [oracle_mod.histogram(x, o, w.BOX_ORTHO, box, 4.0, 90) for x, o in zip(xs, offs)]

    def frames(accumulate, outs, which):
        return [dh.FrameArgs(torch_mod.from_numpy(xs[k]).cuda() if where == "device" else xs[k], offs[k], w.BOX_ORTHO,
                             box, 4.0, 90, outs[k], accumulate) for k in which]

    def fresh():
        if where == "device":
            return [torch_mod.full((3, 90), 5, dtype=torch_mod.int64, device="cuda") for _ in sizes]
        return [np.full((3, 90), 5, dtype=np.uint64) for _ in sizes]

    def values(out):
        return out.cpu().numpy().view(np.uint64) if where == "device" else out

    full = [k for k, n in enumerate(sizes) if n]
    with dh.Context(0) as ctx:
        outs = fresh()
        for _ in range(2):  # (the first call also builds the bin thresholds)
            ctx.histogram_batch(frames(False, outs, full))
        launches = ctx.stats()["kernel_launches"]
        outs = fresh()
        ctx.histogram_batch(frames(False, outs, range(len(sizes))))
        assert ctx.stats()["kernel_launches"] == launches
        for k, out in enumerate(outs):
            assert np.array_equal(values(out), want[k]), k
        ctx.histogram_batch(frames(True, outs, range(len(sizes))))
        for k, out in enumerate(outs):
            assert np.array_equal(values(out), 2 * want[k]), k
        outs = fresh()
        ctx.histogram_batch(frames(False, outs, [0, 2]))  # nothing but empty frames
        assert not values(outs[0]).any() and not values(outs[2]).any()


@pytest.mark.parametrize("box", ["none", "ortho", "triclinic"])
def test_small_species_go_to_the_tiled_kernel(torch_mod, oracle_mod, box):
    # a batch of small frames of eight species (tiled, several to a launch), with one large frame
    # (list kernel) and one beyond half the box among them; outputs overwritten and added to
    rng = w.rng_for(45)
    kinds = {"none": (w.BOX_NONE, lambda s: np.zeros(9)), "ortho": (w.BOX_ORTHO, lambda s: w.ortho_box(s, s, 1.2 * s)),
             "triclinic": (w.BOX_TRICLINIC, lambda s: w.triclinic_box(s, s, s, *w.C3_ANGLES))}
    kind, make = kinds[box]
    frames = []
    for k in range(120):
        n, species = (30_000, 1) if k == 50 else (int(rng.integers(8, 900)), 8)
        side = (n / 0.1) ** (1.0 / 3.0)
        b = make(side)
        m = np.eye(3) * side if box == "none" else w.box_matrix(b)
        r = 1.8 * side if box == "none" else (1.5 if k == 51 else 0.95) * float(w.box_heights(b).min()) / 2.0
        cuts = [n * q // species for q in range(species + 1)]
        frames.append(w.frame_from((rng.random((n, 3)) @ m.T).astype(np.float32), cuts, kind, b, r, 300, str(k)))
    fas = [dh.FrameArgs(torch_mod.from_numpy(f.coords).cuda(), f.offsets, f.box_type, f.box, f.r_max, f.nbins,
                        torch_mod.full((f.n_hist, f.nbins), 3, dtype=torch_mod.int64, device="cuda")) for f in frames]
    with dh.Context(0) as ctx:
        for _ in range(2):
            ctx.histogram_batch(fas)
        assert ctx.stats()["block_threads"] == 256, ctx.stats()  # the tiled kernel's shape
    for fa, f in zip(fas, frames):
        assert np.array_equal(fa.out.cpu().numpy().view(np.uint64), oracle_mod.histogram_frame(f)), f.name


@pytest.mark.parametrize("box", ["none", "ortho"])
def test_one_frame_of_many_species(torch_mod, oracle_mod, box):
    n, species = 2400, 60
    x = (w.rng_for(46).random((n, 3)) * 28.0).astype(np.float32)
    kind, b, r = (w.BOX_NONE, np.zeros(9), 50.0) if box == "none" else (w.BOX_ORTHO, w.ortho_box(28.0), 13.0)
    offs = np.array([n * q // species for q in range(species + 1)], dtype=np.int64)
    want = oracle_mod.histogram(x, offs, kind, b, r, 200)
    dev = torch_mod.from_numpy(x).cuda()
    with dh.Context(0, pool_bytes=256 << 20) as ctx:
        got = ctx.histogram(dev, offs, kind, b, r, 200)
        assert ctx.stats()["block_threads"] == 256, ctx.stats()
        fa = dh.FrameArgs(dev, offs, kind, b, r, 200)
        assert ctx.wait(ctx.submit(fa)) == dh.DH_OK
    assert np.array_equal(got.cpu().numpy().view(np.uint64), want)
    assert torch_mod.equal(fa.out, got)
    few = np.array([n * q // 15 for q in range(16)], dtype=np.int64)  # the allocation-free entry's most
    out = dh.FrameArgs(dev, few, kind, b, r, 200)
    dh.dh_histogram_noalloc(out.frame)
    assert np.array_equal(out.out.cpu().numpy().view(np.uint64), oracle_mod.histogram(x, few, kind, b, r, 200))


@pytest.mark.parametrize("n,species,reach,threads", [(1500, 1, 1.7, 512), (30_000, 1, 1.2, 256), (30_000, 2, 1.7, 256),
                                                     (30_000, 1, 2.2, 256)])
def test_r_max_beyond_half_an_orthorhombic_box(torch_mod, oracle_mod, n, species, reach, threads):
    # the shortest of several images: the list kernel only where a frame is too small for the tiled one
    side = (n / 0.1) ** (1.0 / 3.0)
    f = w.uniform_frame(47, n, w.BOX_ORTHO, w.ortho_box(side, 1.1 * side, side), 0.5 * reach * side, 500,
                        n_species=species)
    dev = torch_mod.from_numpy(f.coords).cuda()
    want = oracle_mod.histogram_frame(f)
    with dh.Context(0, pool_bytes=256 << 20) as ctx:
        got = ctx.histogram(dev, f.offsets, f.box_type, f.box, f.r_max, f.nbins)
        assert ctx.stats()["block_threads"] == threads, ctx.stats()
        fa = dh.FrameArgs(dev, f.offsets, f.box_type, f.box, f.r_max, f.nbins)
        assert ctx.wait(ctx.submit(fa)) == dh.DH_OK
    out = dh.FrameArgs(dev, f.offsets, f.box_type, f.box, f.r_max, f.nbins)
    dh.dh_histogram_noalloc(out.frame)
    for o in (got, fa.out, out.out):
        assert np.array_equal(o.cpu().numpy().view(np.uint64), want)
