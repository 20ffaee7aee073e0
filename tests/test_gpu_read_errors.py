"""Field read-outs after a recorded device error (a persistent launch whose bounded wait ran
out): the error is returned and the caller's array keeps its contents, for every component."""
import ctypes

import numpy as np
import pytest

import paper_0909_5603_gb300 as pic
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()


@pytest.fixture(scope="module")
def failed():
    """The members of a stalled batch that hold a device error."""
    sims, n = [], (48, 1, 40)
    for i in range(3):
        p = synth.random_particles(n, 2, 2000 + 100 * i, 0.2, seed=70 + i)
        s = pic.Simulation(2, n, (0, 0, 0), (1.0, 1.0, 1.0), 0.45, order=2)
        s.load_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
        sims.append(s)
    batch = pic.Batch(sims)
    batch.set_persistent(True, spin_limit=2000, test_stall=1)
    batch.step(2)
    with pytest.raises(pic.PicError) as e:
        batch.synchronize()
    assert e.value.status == pic.PIC_ERR_TIMEOUT
    bad = []
    for s in sims:
        try:
            s.synchronize()
        except pic.PicError:
            bad.append(s)
    assert bad
    yield bad
    batch.close()


@pytest.mark.parametrize("comp", range(pic.PIC_EX, pic.PIC_DIVE + 1))
def test_one_component(failed, comp):
    for s in failed:
        out = np.full(s.ncell, 1234.5)
        assert pic.lib().pic_get_field(s.h, comp, pic._ptr(out), out.size) == pic.PIC_ERR_TIMEOUT
        assert (out == 1234.5).all()


@pytest.mark.parametrize("comps", [[pic.PIC_EX, pic.PIC_BZ, pic.PIC_JY], [pic.PIC_DIVE, pic.PIC_RHO]])
def test_several_components(failed, comps):
    c = (ctypes.c_int * len(comps))(*comps)
    for s in failed:
        out = np.full((len(comps), s.ncell), 1234.5)
        assert pic.lib().pic_get_fields(s.h, c, len(comps), pic._ptr(out), out.size) == pic.PIC_ERR_TIMEOUT
        assert (out == 1234.5).all()
