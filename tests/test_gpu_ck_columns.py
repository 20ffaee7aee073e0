"""The low-dispersion half step of one 3D instance (a thread per column marching along z)
against the per-cell kernel that a batch takes, over column counts and plane counts at and
around a block's columns and a chunk's planes, with mixed boundaries, and full steps after
it.  Both form the same sums in the same order: what can differ is which products are fused."""
import numpy as np
import pytest

import paper_0909_5603_gb300 as pic

pytestmark = pytest.mark.gpu

EB = [pic.PIC_BX, pic.PIC_BY, pic.PIC_BZ, pic.PIC_EX, pic.PIC_EY, pic.PIC_EZ]
CASES = [((8, 8, 8), (0, 0, 0)), ((8, 16, 9), (1, 0, 1)), ((16, 8, 12), (0, 1, 0)), ((33, 9, 26), (0, 1, 1)),
         ((43, 12, 13), (1, 1, 0)), ((160, 128, 97), (1, 0, 0))]


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()


@pytest.mark.parametrize("prec,tol", [(pic.PIC_PREC_FP64, 1e-13), (pic.PIC_PREC_FP32, 2e-6)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("n,bc", CASES)
def test_columns_against_cells(n, bc, prec, tol):
    sims = []
    for _ in range(3):
        s = pic.Simulation(3, n, bc, (1.0, 0.9, 1.1), 0.45, order=1, precision=prec, solver=pic.PIC_SOLVER_CK,
                           absorb_cells=4)
        s.load_particles(np.array([0], np.int32), np.full((1, 3), 0.5), np.zeros((1, 3)), np.zeros(1))
        for c in range(6):
            s.set_field(c, np.random.default_rng(c).standard_normal((n[2], n[1], n[0])))
        sims.append(s)
    alone, batch = sims[0], pic.Batch(sims[1:])
    alone.step(3)
    batch.step(3)
    batch.synchronize()
    for c in EB:
        a, b = alone.get_field(c), sims[1].get_field(c)
        assert np.abs(a - b).max() <= tol * np.abs(b).max(), c
        assert np.array_equal(b, sims[2].get_field(c)), c
    batch.close()
