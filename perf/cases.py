"""Timed cases of the pair-distance histogram library, through its public entry points.

Each case is one call a program makes: a frame (or a batch, a trajectory, a set
of served requests) of N particles in a box type, histogrammed into nbins bins
up to r_max.  Coordinates are uniform at a fixed density or Gaussian clusters on
a uniform background, the two distributions the library's own configurations use.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1808_01478_gb300 as dh

DENSITY = 0.1               # particles per unit volume
ANGLES = (70.0, 80.0, 100.0)  # of the triclinic cell
BOXES = {"none": dh.DH_BOX_NONE, "ortho": dh.DH_BOX_ORTHO, "triclinic": dh.DH_BOX_TRICLINIC}


def _case(name, entry, box, n, bins, species=1, frames=1, dtype="f32", where="device", reach=1.0, clustered=False):
    c = {"entry": entry, "box": box, "n": n, "bins": bins, "species": species, "frames": frames, "dtype": dtype,
         "where": where, "reach": reach, "clustered": clustered}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a small molecule's frame, every pair in range: the latency of one call counts
        _case("small_nobox", "plain", "none", 2000, 1000),
        # a small solvated system read from a file: host arrays in, histograms out, all species pairs
        _case("small_ortho_host", "plain", "ortho", 1501, 1024, species=3, where="host"),
        # the analysis of one frame of a binary solution in a periodic box
        _case("ortho_two_species", "plain", "ortho", 100_000, 10_000, species=2),
        # a crowded solution in a general cell: dense clusters, every species pair, fine bins
        _case("triclinic_clusters", "plain", "triclinic", 500_000, 20_000, species=3, clustered=True),
        # one very large frame of each box type in one batched call
        _case("large_three_boxes", "batch", "mixed", 1_000_000, 10_000, frames=3),
        # a piece of a trajectory with uneven frames in one batched call
        _case("batch_uneven", "batch", "ortho", 50_000, 4096, species=2, frames=64),
        # a binary64 trajectory, so that no input digit is lost
        _case("ortho_f64", "plain", "ortho", 200_001, 8192, species=2, dtype="f64"),
        # a histogram wider than one block's shared memory: several bin sweeps
        _case("ortho_wide", "plain", "ortho", 200_000, 100_000),
        # r_max beyond half the smallest plane spacing: the neighbouring-cell search
        _case("triclinic_search", "plain", "triclinic", 40_000, 4096, species=2, reach=1.6),
        # requests of several users at once, of all sizes and box types
        _case("served_mix", "served", "mixed", 20_000, 4096, species=2, frames=24),
        # a caller that must not allocate device memory
        _case("noalloc_triclinic", "noalloc", "triclinic", 30_011, 8192, species=2),
        # a short trajectory accumulated on the device and normalised to g(r)
        _case("trajectory_rdf", "rdf", "ortho", 6000, 2000, species=2, frames=10),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    entry = rng.choice(["plain", "plain", "plain", "plain", "batch", "served", "noalloc", "rdf"])
    box = rng.choice(["none", "ortho", "triclinic"])
    species = rng.randint(1, 3)
    bins = log_int(500, 20_000)
    clustered = rng.random() < 0.25
    if entry == "plain":
        dtype = rng.choice(["f32", "f32", "f32", "f64"])
        where = rng.choice(["device", "device", "host"])
        if box == "triclinic" and rng.random() < 0.25:
            return _case(None, entry, box, log_int(1000, 60_000), bins, species, 1, dtype, where, 1.6, clustered)
        if rng.random() < 0.2:  # wide histograms: one to several bin sweeps
            return _case(None, entry, box, log_int(20_000, 250_000), log_int(20_000, 120_000), species, 1, dtype,
                         where, 1.0, clustered)
        reach = rng.choice([1.0, 1.0, 0.6])
        return _case(None, entry, box, log_int(1000, 700_000), bins, species, 1, dtype, where, reach, clustered)
    if entry == "batch":
        return _case(None, entry, rng.choice([box, "mixed"]), log_int(5000, 60_000), bins, species, rng.randint(4, 64))
    if entry == "served":
        return _case(None, entry, "mixed", log_int(2000, 40_000), bins, species, rng.randint(4, 32))
    if entry == "noalloc":
        return _case(None, entry, box, log_int(1000, 100_000), bins, species, clustered=clustered)
    return _case(None, entry, box, log_int(1000, 20_000), min(bins, 5000), species, rng.randint(2, 12))


# ----------------------------------------------------------------- inputs


def _box(box, n):
    """Box matrix (rows of a 3x3 whose columns are the box vectors), half its smallest plane spacing (no box: the diagonal)."""
    side = (n / DENSITY) ** (1.0 / 3.0)
    if box != "triclinic":
        return np.diag([side] * 3), side * math.sqrt(3.0) if box == "none" else side / 2.0
    al, be, ga = (math.radians(v) for v in ANGLES)
    cy = (math.cos(al) - math.cos(be) * math.cos(ga)) / math.sin(ga)
    m = np.array([[1.0, math.cos(ga), math.cos(be)], [0.0, math.sin(ga), cy],
                  [0.0, 0.0, math.sqrt(1.0 - math.cos(be) ** 2 - cy ** 2)]])
    m *= (n / DENSITY / np.linalg.det(m)) ** (1.0 / 3.0)
    a, b, c = m.T
    vol = np.linalg.det(m)
    h = min(vol / np.linalg.norm(np.cross(u, v)) for u, v in ((a, b), (b, c), (c, a)))
    return m, 0.95 * h / 2.0


def _sizes(case):
    """Particles and box type of each frame: log-uniform from n / 10 to 4 n where frames are uneven."""
    uneven = case["entry"] == "served" or (case["entry"] == "batch" and case["box"] != "mixed")
    return [(max(64, int(case["n"] * 40.0 ** ((f * 0.6180339887498949) % 1.0) / 10.0)) if uneven else case["n"],
             ("none", "ortho", "triclinic")[f % 3] if case["box"] == "mixed" else case["box"])
            for f in range(case["frames"])]


def _frames(case, seed):
    """The case's frames: coordinates, species offsets, box type, box matrix, r_max."""
    rng = np.random.Generator(np.random.PCG64(seed))
    out = []
    for n, box in _sizes(case):
        m, half = _box(box, n)
        s = rng.random((n, 3))
        if case["clustered"]:
            k = int(0.8 * n)
            width = 2.0 / (n / DENSITY) ** (1.0 / 3.0)
            centres = rng.random((200, 3))
            s[:k] = centres[rng.integers(0, 200, k)] + rng.normal(0.0, width, (k, 3))
            s -= np.floor(s)
            s = s[rng.permutation(n)]
        x = np.ascontiguousarray((m @ s.T).T)
        if case["dtype"] == "f32":
            x = x.astype(np.float32)
        cuts = [0] + [n * (2 * k + 1) // (2 * case["species"]) for k in range(1, case["species"])] + [n]
        out.append((x, np.array(cuts, dtype=np.int64), BOXES[box], np.zeros(9) if box == "none" else m.reshape(9),
                    half * case["reach"]))
    return out


def _pair_densities(offsets, volume):
    n = np.diff(offsets).astype(np.float64)
    return [(n[a] * (n[a] - 1) / 2 if a == b else n[a] * n[b]) / volume
            for a in range(len(n)) for b in range(a, len(n))]


def prepare(case, seed):
    frames = _frames(case, seed)
    if case["where"] == "device":
        frames = [(torch.from_numpy(f[0]).cuda(),) + f[1:] for f in frames]
    hists = dh.n_hist(case["species"])
    outs = [torch.zeros((hists, case["bins"]), dtype=torch.int64, device="cuda") if case["where"] == "device"
            else np.zeros((hists, case["bins"]), dtype=np.uint64) for _ in frames]
    state = {"case": case, "frames": frames, "outs": outs}
    if case["entry"] != "noalloc":
        state["ctx"] = dh.Context(0, pool_bytes=2 << 30)
    if case["entry"] in ("batch", "served", "noalloc"):
        state["args"] = [dh.FrameArgs(x, o, t, b, r, case["bins"], out)
                         for (x, o, t, b, r), out in zip(frames, outs)]
    if case["entry"] == "rdf":
        state["dens"] = _pair_densities(frames[0][1], case["n"] / DENSITY)
    torch.cuda.synchronize()
    return state


def run(state):
    case, frames, outs = state["case"], state["frames"], state["outs"]
    if case["entry"] == "plain":
        x, o, t, b, r = frames[0]
        return state["ctx"].histogram(x, o, t, b, r, case["bins"], outs[0])
    if case["entry"] == "batch":
        state["ctx"].histogram_batch(state["args"])
        return outs
    if case["entry"] == "noalloc":
        dh.dh_histogram_noalloc(state["args"][0].frame)
        return outs[0]
    if case["entry"] == "served":
        tickets = [state["ctx"].submit(a) for a in state["args"]]
        for t in tickets:
            if state["ctx"].wait(t) != dh.DH_OK:
                raise RuntimeError("a request failed")
        return outs
    total = outs[0]
    for k, (x, o, t, b, r) in enumerate(frames):
        state["ctx"].histogram(x, o, t, b, r, case["bins"], total, accumulate=k > 0)
    return {"counts": total, "g": state["ctx"].rdf(total, frames[0][4], state["dens"], len(frames))}


def work(case):
    """Coordinates read and histograms written once; about 10 operations (difference,
    square, sum, root, bin) for each pair within r_max."""
    size = 8 if case["dtype"] == "f64" else 4
    bytes_, flops = 0.0, 0.0
    for n, box in _sizes(case):
        r = _box(box, n)[1] * case["reach"]
        inside = 1.0 if box == "none" else min(1.0, 4.0 / 3.0 * math.pi * r ** 3 / (n / DENSITY))
        bytes_ += 3 * size * n + 8 * dh.n_hist(case["species"]) * case["bins"]
        flops += 10.0 * inside * n * (n - 1) / 2
    return {"bytes": float(bytes_), "flops": float(flops)}


# ----------------------------------------------------------------- 64-bit values


def _counts(x, offsets, box_type, box, r_max, bins):
    """Histograms of one frame in binary64 with plain numpy, in the library's order."""
    x = x.astype(np.float64)
    m = box.reshape(3, 3)
    s = len(offsets) - 1
    out = []
    for a in range(s):
        for b in range(a, s):
            h = np.zeros(bins, dtype=np.int64)
            xb = x[offsets[b]:offsets[b + 1]]
            for i in range(offsets[a], offsets[a + 1]):
                d = (x[i + 1:offsets[a + 1]] if a == b else xb) - x[i]
                if box_type == dh.DH_BOX_ORTHO:
                    d -= np.rint(d * (1.0 / np.diag(m))) * np.diag(m)
                elif box_type == dh.DH_BOX_TRICLINIC:  # r_max below half the smallest plane spacing
                    for q in (2, 1, 0):
                        d -= np.rint(d[:, q] / m[q, q])[:, None] * m[:, q]
                t = bins * np.sqrt((d * d).sum(1)) / r_max
                h += np.bincount(t[t < bins].astype(np.int64), minlength=bins)
            out.append(h)
    return np.stack(out)


def exact(case, seed):
    pairs = case["frames"] * case["n"] ** 2 / 2
    if case["entry"] not in ("plain", "noalloc", "rdf") or pairs > 2.5e8 or case["reach"] > 1.0 and case["box"] != "none":
        return None
    frames = _frames(case, seed)
    total = sum(_counts(x, o, t, b, r, case["bins"]) for x, o, t, b, r in frames)
    if case["entry"] != "rdf":
        return total
    r = frames[0][4]
    edges = np.arange(case["bins"] + 1, dtype=np.float64) * (r / case["bins"])
    shell = 4.0 * math.pi / 3.0 * np.diff(edges ** 3)
    dens = np.array(_pair_densities(frames[0][1], case["n"] / DENSITY))
    return {"counts": total, "g": total / len(frames) / (dens[:, None] * shell[None, :])}
