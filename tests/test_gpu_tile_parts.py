"""Crowded tiles in parts, at the edges of a split, for both least sizes of a part: parts of
eight chunks of 256 particles in grids of at least 304 tiles in FP32 (a tile of 16 chunks is
taken whole, one particle more splits it), and parts of one chunk in smaller grids and in
FP64 (2 chunks whole, 3 in parts).  Against the FP64 oracle over three particle phases, which
the next phase and the read-out find through the parts' joined chunk records: FP32 the
current normwise within 2e-6, the bar of the block-scaled accumulation, and the momenta;
FP64 1e-12 with the canonical order and the cells bit for bit."""
import numpy as np
import pytest

import oracle
import paper_0909_5603_gb300 as pic
import synth

pytestmark = pytest.mark.gpu

FP32, FP64 = pic.PIC_PREC_FP32, pic.PIC_PREC_FP64
JS = [pic.PIC_JX, pic.PIC_JY, pic.PIC_JZ]
DT = 0.45
LARGE = {3: ((56, 56, 56), 8), 2: ((288, 1, 304), 16)}  # 343 and 342 tiles
SMALL = {3: ((24, 24, 24), 8), 2: ((48, 1, 48), 16)}    # 27 and 9


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()
    oracle.build()


def crowds(ndim, n, ts, counts, seed):
    """counts[m] particles in tile m of a few tiles (two neighbours and the box's corners), one
    in each of some others."""
    rng = np.random.default_rng(seed)
    last = [(n[a] - 1) // ts for a in range(3)]
    tiles = [(1, 1, 1), (2, 1, 1), (0, 0, 0), (last[0], last[1], last[2])]
    at = [rng.integers(0, ts, (c, 3)) + ts * np.array(t) for c, t in zip(counts, tiles)]
    at.append(rng.integers(0, np.array(n), (50, 3)))
    at = np.concatenate(at)
    if ndim == 2:
        at[:, 1] = 0
    m = len(at)
    order = rng.permutation(m)  # as a user's arrays: not sorted by tile
    at = at[order]
    off = synth.f32(rng.random((m, 3), dtype=np.float32))
    if ndim == 2:
        off[:, 1] = 0.0
    return dict(cell=(at[:, 0] + n[0] * (at[:, 1] + n[1] * at[:, 2])).astype(np.int32), off=off,
                u=synth.f32(rng.normal(0.0, 0.8, (m, 3))), w=synth.f32(rng.uniform(0.5, 1.5, m)),
                id=np.arange(m, dtype=np.int32))


def run(ndim, grid, bc, order, prec, counts, seed):
    n, ts = grid
    fields = synth.smooth_fields(n, ndim, 0.2, seed=seed)
    p = crowds(ndim, n, ts, counts, seed + 1)
    o = oracle.Sim(ndim, n, bc, (1.0, 1.0, 1.0), DT, order=order, tile=(ts, ts if ndim == 3 else 1, ts))
    g = pic.Simulation(ndim, n, bc, (1.0, 1.0, 1.0), DT, order=order, precision=prec)
    for c, f in enumerate(fields):
        o.set_field(c, f)
        g.set_field(c, f)
    o.set_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
    g.load_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
    tol = 2e-6 if prec == FP32 else 1e-12
    for _ in range(3):
        g.run_phases(pic.PIC_PHASE_PARTICLES)
        o.particle_phase()
        for c in JS:
            jg, jo = g.get_field(c), o.get_field(c)
            assert np.linalg.norm(jg - jo) <= tol * np.linalg.norm(jo), c
        pg, po = g.get_particles(), o.get_particles()
        if prec == FP64:
            assert np.array_equal(pg["id"], po["id"]) and np.array_equal(pg["cell"], po["cell"])
        # (FP32: a particle within a rounding of an absorbing face may stay on one side only)
        ids, ig, io = np.intersect1d(pg["id"], po["id"], return_indices=True)
        assert max(pg["id"].size, po["id"].size) - ids.size <= (0 if prec == FP64 or 1 not in bc else 2)
        assert np.linalg.norm(pg["u"][ig] - po["u"][io]) <= tol * np.linalg.norm(po["u"][io])


@pytest.mark.parametrize("counts", [(16 * 256, 0, 0, 0), (16 * 256 + 1, 0, 0, 0), (24 * 256, 24 * 256 + 1, 0, 0),
                                    (17 * 256 + 5, 16 * 256, 0, 40 * 256 + 131), (9000, 4097, 12000, 5000)])
@pytest.mark.parametrize("ndim,order,bc", [(3, 2, (0, 0, 0)), (3, 1, (1, 0, 1)), (2, 2, (0, 0, 0)), (2, 1, (1, 0, 0))])
def test_parts_of_eight_chunks(ndim, order, bc, counts):
    run(ndim, LARGE[ndim], bc, order, FP32, counts, 500 + counts[0])


@pytest.mark.parametrize("counts", [(2 * 256, 0, 0, 0), (2 * 256 + 1, 0, 0, 0), (3 * 256, 3 * 256 + 1, 0, 0),
                                    (700, 513, 1300, 512)])
@pytest.mark.parametrize("ndim,order,prec", [(3, 2, FP32), (2, 2, FP32), (2, 1, FP32), (3, 2, FP64), (2, 1, FP64)])
def test_parts_of_one_chunk(ndim, order, prec, counts):
    run(ndim, SMALL[ndim], (0, 0, 0), order, prec, counts, 600 + counts[0])


@pytest.mark.parametrize("ndim,order", [(3, 2), (2, 2)])
def test_parts_of_one_chunk_in_a_large_fp64_grid(ndim, order):
    run(ndim, LARGE[ndim], (0, 0, 0), order, FP64, (1000, 513, 700, 300), 700)
