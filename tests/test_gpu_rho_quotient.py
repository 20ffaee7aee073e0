"""The density of single particles on nodes is their charge divided by the cell volume,
correctly rounded: order 1, one particle on each of some distant nodes, so that every
deposited value is one quotient, bit for bit as FP64 numpy forms it."""
import numpy as np
import pytest

import paper_0909_5603_gb300 as pic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()


@pytest.mark.parametrize("prec", [pic.PIC_PREC_FP32, pic.PIC_PREC_FP64], ids=["fp32", "fp64"])
@pytest.mark.parametrize("ndim,n,dx", [(3, (12, 16, 24), (2.0, 2.0, 13.0 * (1.0 + (1.0 - 1.0 / 169.0) ** 0.5) / 16.0)),
                                       (3, (16, 8, 32), (0.9, 1.1, 0.7)), (2, (40, 1, 32), (0.3, 1.0, 0.0371))])
def test_one_quotient_per_particle(ndim, n, dx, prec):
    rng = np.random.default_rng(6)
    cells = [i + n[0] * (j + n[1] * k) for k in range(0, n[2], 4) for j in range(0, n[1], 4) for i in range(0, n[0], 4)]
    cell = np.array(cells, np.int32)
    w = rng.uniform(0.1, 2.0, cell.size).astype(np.float32).astype(np.float64)
    charge = -1.6
    s = pic.Simulation(ndim, n, (0, 0, 0), dx, 0.3 * min(dx), precision=prec, order=1, charge=charge)
    s.load_particles(cell, np.zeros((cell.size, 3)), np.zeros((cell.size, 3)), w)
    want = np.zeros(n[0] * n[1] * n[2])
    want[cell] = charge * w / (dx[0] * dx[1] * dx[2])
    assert np.array_equal(s.get_field(pic.PIC_RHO).reshape(-1), want)
