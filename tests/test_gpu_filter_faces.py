"""The fixed-pass current filter at absorbing faces, where it convolves the odd reflection of
the field instead of running the passes: axes from the shortest (8 cells, 4 passes reach the
middle from both faces) to one and more pencils of 64 with remainders, against the FP64
oracle's pass by pass filter.  FP64 1e-14 normwise (sums of at most 9 terms per axis), FP32
1e-6."""
import numpy as np
import pytest

import oracle
import paper_0909_5603_gb300 as pic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()
    oracle.build()


@pytest.mark.parametrize("prec,tol", [(pic.PIC_PREC_FP64, 1e-14), (pic.PIC_PREC_FP32, 1e-6)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("passes", [1, 2, 3, 4])
@pytest.mark.parametrize("ndim,n,bc", [(3, (8, 9, 10), (1, 1, 1)), (3, (65, 8, 13), (1, 0, 1)), (3, (12, 70, 9), (0, 1, 1)),
                                       (3, (9, 8, 131), (1, 1, 1)), (2, (63, 1, 64), (1, 0, 1)), (2, (130, 1, 66), (0, 0, 1))])
def test_filter_at_faces(ndim, n, bc, passes, prec, tol):
    g = pic.Simulation(ndim, n, bc, (1.0, 1.0, 1.0), 0.3, precision=prec, filter_passes=passes)
    o = oracle.Sim(ndim, n, bc, (1.0, 1.0, 1.0), 0.3, filter_passes=passes, tile=(8, 8, 8) if ndim == 3 else (16, 1, 16))
    g.load_particles(np.zeros(0, np.int32), np.zeros((0, 3)), np.zeros((0, 3)), np.zeros(0))
    rng = np.random.default_rng(10 + passes)
    for c in (pic.PIC_JX, pic.PIC_JY, pic.PIC_JZ):
        f = rng.normal(size=(n[2], n[1], n[0])).astype(np.float32).astype(np.float64)
        g.set_field(c, f)
        o.set_field(c, f)
    g.run_phases(pic.PIC_PHASE_FILTER)
    o.filter()
    for c in (pic.PIC_JX, pic.PIC_JY, pic.PIC_JZ):
        a, b = g.get_field(c), o.get_field(c)
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), c
        assert np.abs(a - b).max() <= 10 * tol * np.abs(b).max(), c
