"""The fused Yee update over its tiles and z chunks, against the FP64 oracle (1e-12, full
steps, so that the gather reads the periodic images the update stores in the ghost layers):
grids below, at and just above what a block puts out (29 x 13 columns in 3D, strips of 29 in
2D3V) and a ghost width
(cells that are images beyond both faces of a periodic axis), mixed boundaries, alone and
as members of a batch."""
import numpy as np
import pytest

import oracle
import paper_0909_5603_gb300 as pic
import synth

pytestmark = pytest.mark.gpu

FIELDS = [pic.PIC_EX, pic.PIC_EY, pic.PIC_EZ, pic.PIC_BX, pic.PIC_BY, pic.PIC_BZ]
DT = 0.45
GRIDS = {
    3: [((8, 8, 8), (0, 0, 0)), ((8, 24, 33), (0, 0, 0)), ((33, 9, 26), (0, 1, 0)), ((64, 8, 40), (1, 0, 1)),
        ((31, 25, 70), (0, 0, 1)), ((29, 13, 24), (1, 1, 0)), ((30, 14, 24), (1, 0, 0)), ((58, 27, 9), (0, 0, 1))],
    2: [((16, 1, 16), (0, 0, 0)), ((64, 1, 49), (0, 0, 0)), ((65, 1, 130), (0, 0, 1)), ((130, 1, 48), (1, 0, 0)), ((29, 1, 48), (1, 0, 0)),
        ((59, 1, 50), (0, 0, 0))],
}


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()
    oracle.build()


def pair(ndim, n, bc, prec, seed):
    ts = (8, 8, 8) if ndim == 3 else (16, 1, 16)
    g = pic.Simulation(ndim, n, bc, (1.0, 1.0, 1.0), DT, order=2, precision=prec, absorb_cells=4)
    o = oracle.Sim(ndim, n, bc, (1.0, 1.0, 1.0), DT, order=2, tile=ts, absorb_cells=4)
    for c, f in enumerate(synth.smooth_fields(n, ndim, 0.2, seed=seed)):
        g.set_field(c, f)
        o.set_field(c, f)
    p = synth.random_particles(n, ndim, 3000, 0.5, seed=seed + 1)
    g.load_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
    o.set_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
    return g, o


def check(g, o, tol):
    for c in FIELDS:
        a, b = g.get_field(c), o.get_field(c)
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), c


@pytest.mark.parametrize("ndim,n,bc", [(d, n, bc) for d in (3, 2) for n, bc in GRIDS[d]])
@pytest.mark.parametrize("prec,tol", [(pic.PIC_PREC_FP64, 1e-12), (pic.PIC_PREC_FP32, 1e-5)], ids=["fp64", "fp32"])
def test_full_steps_over_tile_edges(ndim, n, bc, prec, tol):
    g, o = pair(ndim, n, bc, prec, 31)
    g.step(5)
    o.step(5)
    check(g, o, tol)


@pytest.mark.parametrize("ndim", [3, 2])
def test_batch_of_uneven_grids(ndim):
    pairs = [pair(ndim, n, bc, pic.PIC_PREC_FP64, 41 + k) for k, (n, bc) in enumerate(GRIDS[ndim])]
    batch = pic.Batch([g for g, _ in pairs])
    batch.step(4)
    batch.synchronize()
    for g, o in pairs:
        o.step(4)
        check(g, o, 1e-12)
        g.step(2)  # alone again: its own chunks of the update
        o.step(2)
        check(g, o, 1e-12)
