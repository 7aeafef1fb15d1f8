"""The list kernel (runs of 128 particles against listed particle images) at the
sizes where it can go wrong, bin for bin against the FP64 oracle: runs one short
and one over, species of one run and of several, several bin sweeps, r_max of
exactly half the box (two images of a pair on the last edge), coordinates in
several cells and far off the origin, lattices on the bin edges, and particles at
the same place.  Integer counts: no tolerance.
"""
import numpy as np
import pytest

import paper_1808_01478_gb300 as dh
import workloads as w

pytestmark = pytest.mark.gpu

BOX = {"none": (w.BOX_NONE, np.zeros(9)), "ortho": (w.BOX_ORTHO, w.ortho_box(21.0, 17.0, 26.0)),
       "tric": (w.BOX_TRICLINIC, w.triclinic_box(20, 19, 23, *w.C3_ANGLES))}


def half(kind):
    return float(w.box_heights(BOX[kind][1]).min()) / 2.0


def check(oracle_mod, x, offs, kind, r_max, nbins):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    box_type, box = BOX[kind]
    x = np.ascontiguousarray(x)
    want = oracle_mod.histogram(x, np.asarray(offs, np.int64), box_type, box, r_max, nbins)
    with dh.Context(0) as ctx:
        got = ctx.histogram(torch.from_numpy(x).cuda(), offs, box_type, box, r_max, nbins)
        # again: workspaces reused
        again = ctx.histogram(torch.from_numpy(x).cuda(), offs, box_type, box, r_max, nbins)
    got, again = got.cpu().numpy().view(np.uint64), again.cpu().numpy().view(np.uint64)
    bad = np.argwhere(got != want)
    assert bad.size == 0, (len(bad), bad[:4].tolist())
    assert np.array_equal(got, again)


def uniform(kind, n, seed):
    box = BOX[kind][1] if kind != "none" else w.ortho_box(20.0)
    return w.uniform_in_cell(w.rng_for(seed), n, box)


@pytest.mark.parametrize("kind", ["none", "ortho", "tric"])
@pytest.mark.parametrize("sizes", [[1], [2], [127], [128], [129], [257], [1, 128], [129, 0, 31], [640, 5], [3000, 129]],
                         ids=lambda s: "-".join(map(str, s)))
def test_run_boundaries(oracle_mod, kind, sizes):
    offs = np.concatenate([[0], np.cumsum(sizes)])
    x = uniform(kind, int(offs[-1]), 11)
    r = 25.0 if kind == "none" else half(kind) * (1.0 if kind == "ortho" else 0.97)
    check(oracle_mod, x, offs, kind, r, 701)


@pytest.mark.parametrize("kind", ["none", "ortho", "tric"])
@pytest.mark.parametrize("nbins,reach", [(1, 0.9), (7, 0.3), (40_000, 0.9), (34_900, 0.6), (130_000, 0.97)])
def test_bins_and_sweeps(oracle_mod, kind, nbins, reach):
    x = uniform(kind, 2500, 12)
    check(oracle_mod, x, [0, 900, 2500], kind, reach * (34.0 if kind == "none" else half(kind)), nbins)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("kind,cells", [("ortho", 2), ("tric", 3), ("ortho", 700), ("tric", 100_000), ("tric", 3_000_000)])
def test_particles_in_several_cells(oracle_mod, kind, cells, dtype):
    rng = w.rng_for(13)
    m = w.box_matrix(BOX[kind][1])
    x = (m @ rng.random((700, 3)).T).T + rng.integers(-cells, cells + 1, (700, 3)).astype(np.float64) @ m.T
    check(oracle_mod, x.astype(dtype), [0, 300, 700], kind, 0.95 * half(kind), 500)


@pytest.mark.parametrize("kind", ["none", "ortho", "tric"])
def test_far_from_the_origin(oracle_mod, kind):
    x = (uniform(kind, 900, 14).astype(np.float64) + 3.0e5).astype(np.float32)
    check(oracle_mod, x, [0, 900], kind, 9.0 if kind == "none" else 0.95 * half(kind), 300)


def test_half_box_lattice_and_coincident_particles(oracle_mod):
    # an integer lattice in a box of side 16, r_max = L/2 on the last edge; half of
    # the particles twice, so pairs at distance 0 as well
    BOX["lattice"] = (w.BOX_ORTHO, w.ortho_box(16.0))
    g = np.arange(16, dtype=np.float32)
    x = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)[::7]
    x = np.concatenate([x, x[::2]]).copy()
    for nbins in (8, 16, 1024):
        check(oracle_mod, x, [0, 400, len(x)], "lattice", 8.0, nbins)


@pytest.mark.parametrize("sizes", [[1, 128], [129, 0, 31], [640, 5], [3000, 129]], ids=lambda s: "-".join(map(str, s)))
@pytest.mark.parametrize("kind,reach", [("ortho", 1.02), ("ortho", 1.7), ("ortho", 4.0), ("tric", 1.0), ("tric", 1.6),
                                        ("tric", 3.0)])
def test_r_max_beyond_half_the_image_distance(oracle_mod, kind, reach, sizes):
    # several images of a pair inside r_max: the shortest counts
    offs = np.concatenate([[0], np.cumsum(sizes)])
    check(oracle_mod, uniform(kind, int(offs[-1]), 15), offs, kind, reach * half(kind), 801)


@pytest.mark.parametrize("kind", ["ortho", "tric"])
@pytest.mark.parametrize("nbins", [2, 50_000, 110_000])
def test_shortest_image_over_sweeps_and_cells(oracle_mod, kind, nbins):
    rng = w.rng_for(16)
    m = w.box_matrix(BOX[kind][1])
    x = (m @ rng.random((900, 3)).T).T + rng.integers(-3, 4, (900, 3)).astype(np.float64) @ m.T
    check(oracle_mod, x.astype(np.float32), [0, 350, 900], kind, 1.5 * half(kind), nbins)


def test_cells_whose_27_images_can_miss_the_shortest(oracle_mod):
    # a flat cell: the definition's minimum over 27 shifts is not the lattice's
    BOX["flat"] = (w.BOX_TRICLINIC, np.array([10.0, 4.0, 4.9, 0.0, 9.0, 4.4, 0.0, 0.0, 2.0]))
    x = w.uniform_in_cell(w.rng_for(17), 600, BOX["flat"][1])
    check(oracle_mod, x, [0, 200, 600], "flat", 5.0, 300)
