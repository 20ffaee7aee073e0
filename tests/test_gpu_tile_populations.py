"""The particle phase over tile populations at the edges of a chunk of 256 particles (a
warp, a chunk, several chunks, each with a remainder): one crowded tile next to empty
ones, and tiles crowded enough to be worked on in parts by several CTAs, against the FP64 oracle, for one instance and for a batch.  FP32 after one phase:
J normwise within 2e-6, the bar of the block-scaled accumulation; FP64: 1e-12."""
import numpy as np
import pytest

import oracle
import paper_0909_5603_gb300 as pic
import synth

pytestmark = pytest.mark.gpu

FP32, FP64 = pic.PIC_PREC_FP32, pic.PIC_PREC_FP64
JS = [pic.PIC_JX, pic.PIC_JY, pic.PIC_JZ]
GRID = {3: ((24, 24, 24), 8), 2: ((48, 1, 48), 16)}
DT = 0.45


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()
    oracle.build()


def crowd(ndim, count, seed):
    """`count` particles of tile (1, 1, 1) and one in the tile beside it."""
    n, ts = GRID[ndim]
    rng = np.random.default_rng(seed)
    at = rng.integers(ts, 2 * ts, (count + 1, 3))
    at[-1] = ts - 1
    if ndim == 2:
        at[:, 1] = 0
    cell = (at[:, 0] + n[0] * (at[:, 1] + n[1] * at[:, 2])).astype(np.int32)
    off = synth.f32(rng.random((count + 1, 3), dtype=np.float32))
    if ndim == 2:
        off[:, 1] = 0.0
    u = synth.f32(rng.normal(0.0, 0.8, (count + 1, 3)))
    w = synth.f32(rng.uniform(0.5, 1.5, count + 1))
    return dict(cell=cell, off=off, u=u, w=w, id=np.arange(count + 1, dtype=np.int32))


def make(ndim, order, prec, parts, fields):
    n, ts = GRID[ndim]
    g = pic.Simulation(ndim, n, (0, 0, 0), (1.0, 1.0, 1.0), DT, order=order, precision=prec)
    for c, f in enumerate(fields):
        g.set_field(c, f)
    g.load_particles(parts["cell"], parts["off"], parts["u"], parts["w"], parts["id"])
    return g


def check(g, o, prec, ndim):
    tol = 2e-6 if prec == FP32 else 1e-12
    for c in JS:
        jg, jo = g.get_field(c), o.get_field(c)
        assert np.linalg.norm(jg - jo) <= tol * np.linalg.norm(jo), c
    pg, po = g.get_particles(), o.get_particles()
    if prec == FP64:
        assert np.array_equal(pg["id"], po["id"]) and np.array_equal(pg["cell"], po["cell"])
    ig, io = np.argsort(pg["id"]), np.argsort(po["id"])
    assert np.array_equal(pg["id"][ig], po["id"][io])
    assert np.linalg.norm(pg["u"][ig] - po["u"][io]) <= tol * np.linalg.norm(po["u"])


@pytest.mark.parametrize("count", [1, 31, 33, 255, 256, 257, 513, 1024, 1300])
@pytest.mark.parametrize("ndim,order,prec", [(3, 2, FP32), (3, 1, FP32), (2, 2, FP32), (3, 2, FP64), (2, 1, FP64)])
def test_populations_around_a_chunk(ndim, order, prec, count):
    n, ts = GRID[ndim]
    fields = synth.smooth_fields(n, ndim, 0.2, seed=21)
    parts = [crowd(ndim, count, 100 + count), crowd(ndim, max(1, count - 1), 200 + count)]
    oracles = []
    for p in parts:
        o = oracle.Sim(ndim, n, (0, 0, 0), (1.0, 1.0, 1.0), DT, order=order, tile=(ts, ts if ndim == 3 else 1, ts))
        for c, f in enumerate(fields):
            o.set_field(c, f)
        o.set_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
        o.particle_phase()
        oracles.append(o)
    alone = make(ndim, order, prec, parts[0], fields)
    alone.run_phases(pic.PIC_PHASE_PARTICLES)
    check(alone, oracles[0], prec, ndim)
    members = [make(ndim, order, prec, p, fields) for p in parts]
    batch = pic.Batch(members)
    pic.pic_run_phases(batch.h, pic.PIC_PHASE_PARTICLES)
    batch.synchronize()
    for m, o in zip(members, oracles):
        check(m, o, prec, ndim)


@pytest.mark.parametrize("count", [16 * 256, 16 * 256 + 1, 24 * 256, 9000])
@pytest.mark.parametrize("ndim,order,prec", [(3, 2, FP32), (2, 2, FP32), (3, 1, FP64), (2, 2, FP64)])
def test_crowded_tile_in_parts(ndim, order, prec, count):
    """A tile of 16 chunks (the most that one CTA takes whole here), one particle more, and
    further multiples of a part: three phases keep the canonical order (FP64: bit for bit),
    which the next phase and the read-out find through the parts' joined chunk records."""
    n, ts = GRID[ndim]
    fields = synth.smooth_fields(n, ndim, 0.2, seed=22)
    p = crowd(ndim, count, 300 + count)
    o = oracle.Sim(ndim, n, (0, 0, 0), (1.0, 1.0, 1.0), DT, order=order, tile=(ts, ts if ndim == 3 else 1, ts))
    for c, f in enumerate(fields):
        o.set_field(c, f)
    o.set_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
    g = make(ndim, order, prec, p, fields)
    for _ in range(3):
        g.run_phases(pic.PIC_PHASE_PARTICLES)
        o.particle_phase()
        check(g, o, prec, ndim)
