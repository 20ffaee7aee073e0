"""The node divergence of E as the sum of the axes' quotients, each correctly rounded: the
same bits as FP64 numpy forms from the stored fields, for spacings that are no powers of
two, boundaries of both kinds, 2D3V and 3D and both storage precisions."""
import numpy as np
import pytest

import paper_0909_5603_gb300 as pic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()


def below(f, axis, periodic):
    """The value one cell below along a numpy axis: wrapped, or zero beyond the face."""
    g = np.roll(f, 1, axis)
    if not periodic:
        np.moveaxis(g, axis, 0)[0] = 0.0
    return g


@pytest.mark.parametrize("prec", [pic.PIC_PREC_FP32, pic.PIC_PREC_FP64], ids=["fp32", "fp64"])
@pytest.mark.parametrize("ndim,n,bc,dx", [(3, (13, 9, 21), (0, 1, 0), (0.9, 1.1, 0.7)),
                                          (3, (32, 16, 24), (1, 0, 1), (2.0, 2.0, 13.0 / 15.0)),
                                          (2, (37, 1, 26), (0, 0, 1), (0.3, 1.0, 0.0371))])
def test_quotients_bit_for_bit(ndim, n, bc, dx, prec):
    s = pic.Simulation(ndim, n, bc, dx, 0.3 * min(dx), precision=prec)
    rng = np.random.default_rng(5)
    for c in range(3):
        s.set_field(c, rng.standard_normal((n[2], n[1], n[0])))
    want = np.zeros((n[2], n[1], n[0]))
    for a in range(3):
        if ndim == 2 and a == 1:
            continue
        e = s.get_field(a)
        want = want + (e - below(e, 2 - a, bc[a] == 0)) / dx[a]
    assert np.array_equal(s.get_field(pic.PIC_DIVE), want)
