"""The fused Yee update on grids whose z chunks are long (the ring of planes ahead is reused
several times) and end in a shorter one, with the periodic images stored, against the FP64
oracle over full steps: bars as for the short chunks (1e-12 in FP64, 1e-5 in FP32).  That
the library takes the chunks named here is checked by test_maxwell_chunks.py."""
import numpy as np
import pytest

import oracle
import paper_0909_5603_gb300 as pic
import synth

pytestmark = pytest.mark.gpu

FP32, FP64 = pic.PIC_PREC_FP32, pic.PIC_PREC_FP64
FIELDS = [pic.PIC_EX, pic.PIC_EY, pic.PIC_EZ, pic.PIC_BX, pic.PIC_BY, pic.PIC_BZ]
DT = 0.45
# grid, boundaries, planes per chunk in FP64 and FP32
CASES = [(3, (145, 130, 37), (0, 0, 0), 13, 7), (3, (146, 129, 53), (1, 0, 0), 11, 11),
         (3, (203, 92, 51), (0, 1, 1), 26, 11), (2, (290, 1, 2003), (0, 0, 0), 9, 5), (2, (609, 1, 1500), (1, 0, 0), 14, 7)]


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()
    oracle.build()


@pytest.mark.parametrize("prec,tol", [(FP64, 1e-12), (FP32, 1e-5)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("ndim,n,bc,p64,p32", CASES)
def test_full_steps_over_long_chunks(ndim, n, bc, p64, p32, prec, tol):
    assert n[2] % (p64 if prec == FP64 else p32) != 0
    ts = (8, 8, 8) if ndim == 3 else (16, 1, 16)
    g = pic.Simulation(ndim, n, bc, (1.0, 1.0, 1.0), DT, order=2, precision=prec, absorb_cells=4)
    o = oracle.Sim(ndim, n, bc, (1.0, 1.0, 1.0), DT, order=2, tile=ts, absorb_cells=4)
    for c, f in enumerate(synth.smooth_fields(n, ndim, 0.2, seed=61)):
        g.set_field(c, f)
        o.set_field(c, f)
    p = synth.random_particles(n, ndim, 20000, 0.5, seed=62)
    g.load_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
    o.set_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
    g.step(4)
    o.step(4)
    for c in FIELDS:
        a, b = g.get_field(c), o.get_field(c)
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), c
        # plane by plane too: a wrong plane at the end of one chunk would drown in the norm
        d = np.sqrt(((a - b) ** 2).sum((1, 2)))
        assert d.max() <= 10 * tol * np.sqrt((b ** 2).sum((1, 2))).max(), c
    pg, po = g.get_particles(), o.get_particles()
    _, ig, io = np.intersect1d(pg["id"], po["id"], return_indices=True)
    assert ig.size >= 0.9 * pg["id"].size
    assert np.linalg.norm(pg["u"][ig] - po["u"][io]) <= tol * np.linalg.norm(po["u"][io])
