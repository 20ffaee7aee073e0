"""The low-dispersion half step of one 3D FP32 instance on grids whose z chunks have several
planes (the planes of the march are handed on) and whose columns do not fill their last
block, with every kind of boundary along z, against a batch, whose members take the cell
kernel: the same sums in the same order, so that only fused products can differ (2e-6, the
bar of the short chunks), and against the FP64 oracle (1e-5)."""
import numpy as np
import pytest

import oracle
import paper_0909_5603_gb300 as pic

pytestmark = pytest.mark.gpu

EB = [pic.PIC_EX, pic.PIC_EY, pic.PIC_EZ, pic.PIC_BX, pic.PIC_BY, pic.PIC_BZ]
# grid, boundaries, planes per chunk: columns of 128 in blocks, chunks to fill 608 blocks
CASES = [((161, 127, 97), (0, 1, 0), 14), ((203, 101, 40), (0, 0, 1), 14), ((333, 100, 33), (1, 0, 0), 17),
         ((99, 401, 45), (0, 0, 0), 15)]


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()
    oracle.build()


def chunk_planes(n):
    up = lambda a, b: -(-a // b)
    cols = up(n[0] * n[1], 128)
    waves = up(cols * up(n[2], 32), 608)
    return up(n[2], max(1, 608 * waves // cols))


@pytest.mark.parametrize("n,bc,planes", CASES)
def test_march_against_cells_and_oracle(n, bc, planes):
    assert chunk_planes(n) == planes > 2 and (n[0] * n[1]) % 128 != 0
    rng = np.random.default_rng(9)
    fields = [rng.standard_normal((n[2], n[1], n[0])) for _ in range(6)]
    sims = []
    for _ in range(2):
        s = pic.Simulation(3, n, bc, (1.0, 0.9, 1.1), 0.45, order=1, solver=pic.PIC_SOLVER_CK, absorb_cells=4)
        s.load_particles(np.array([0], np.int32), np.full((1, 3), 0.5), np.zeros((1, 3)), np.zeros(1))
        for c in range(6):
            s.set_field(c, fields[c])
        sims.append(s)
    o = oracle.Sim(3, n, bc, (1.0, 0.9, 1.1), 0.45, order=1, solver=1, absorb_cells=4)
    o.set_particles(np.array([0], np.int32), np.full((1, 3), 0.5), np.zeros((1, 3)), np.zeros(1))
    for c in range(6):
        o.set_field(c, fields[c])
    batch = pic.Batch(sims[1:])
    sims[0].step(3)
    batch.step(3)
    batch.synchronize()
    o.step(3)
    for c in EB:
        a, b, w = sims[0].get_field(c), sims[1].get_field(c), o.get_field(c)
        assert np.abs(a - b).max() <= 2e-6 * np.abs(b).max(), c
        assert np.linalg.norm(a - w) <= 1e-5 * np.linalg.norm(w), c
    batch.close()
