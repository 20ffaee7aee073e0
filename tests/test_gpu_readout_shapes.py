"""The density, the Gauss residual and the diagnostics, which walk the particle chunks by
warps, over layouts where the walk can go wrong: one tile, empty tiles at either end, one
crowded tile, more tiles than particles, 2D3V; and several components in one read against
one by one.  FP64, against the oracle: 1e-12 of the largest value (the same terms, summed in
another order)."""
import numpy as np
import pytest

import oracle
import paper_0909_5603_gb300 as pic
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    pic.build()
    oracle.build()


def particles(ndim, n, where, count, seed):
    rng = np.random.default_rng(seed)
    lo, hi = where
    at = np.stack([rng.integers(min(lo, m - 1), min(hi, m), count) for m in n], 1)
    cell = (at[:, 0] + n[0] * (at[:, 1] + n[1] * at[:, 2])).astype(np.int32)
    off = synth.f32(rng.random((count, 3), dtype=np.float32))
    if ndim == 2:
        off[:, 1] = 0.0
    return dict(cell=cell, off=off, u=synth.f32(rng.normal(0.0, 0.5, (count, 3))), w=synth.f32(rng.uniform(0.5, 1.5, count)),
                id=np.arange(count, dtype=np.int32))


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("ndim,n,bc,where,count", [
    (3, (8, 8, 8), (0, 0, 0), (0, 8), 700),         # a single tile
    (3, (32, 24, 40), (0, 1, 0), (24, 40), 257),    # the first tiles empty
    (3, (24, 24, 24), (1, 1, 1), (0, 8), 9000),     # one crowded tile, the others empty
    (3, (48, 48, 48), (0, 0, 0), (0, 48), 40),      # 216 tiles, 40 particles
    (2, (48, 1, 80), (1, 0, 0), (0, 80), 3000),
])
def test_density_and_sums(ndim, n, bc, where, count, order):
    ts = (8, 8, 8) if ndim == 3 else (16, 1, 16)
    p = particles(ndim, n, where, count, 50 + count)
    g = pic.Simulation(ndim, n, bc, (1.0, 0.9, 1.1), 0.4, order=order, precision=pic.PIC_PREC_FP64)
    o = oracle.Sim(ndim, n, bc, (1.0, 0.9, 1.1), 0.4, order=order, tile=ts)
    for c, f in enumerate(synth.smooth_fields(n, ndim, 0.1, seed=51)):
        g.set_field(c, f)
        o.set_field(c, f)
    g.load_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
    o.set_particles(p["cell"], p["off"], p["u"], p["w"], p["id"])
    for steps in (0, 2):
        g.step(steps)
        o.step(steps)
        rho, div = o.rho(), o.div_e()
        got = g.get_fields([pic.PIC_RHO, pic.PIC_EX, pic.PIC_DIVE, pic.PIC_BZ])
        assert np.abs(got[0] - rho).max() <= 1e-12 * np.abs(rho).max()
        assert np.abs(got[2] - div).max() <= 1e-12 * np.abs(div).max()
        assert np.array_equal(got[1], g.get_field(pic.PIC_EX)) and np.array_equal(got[3], g.get_field(pic.PIC_BZ))
        gap = np.abs(div - rho)
        assert abs(g.gauss_residual()[0] - gap.max()) <= 1e-11 * max(np.abs(rho).max(), np.abs(div).max())
        dg, do = g.diagnostics(), o.diagnostics()
        assert dg["n_particles"] == do["n_particles"] == g.num_particles() and dg["n_lost"] == do["n_lost"]
        for k in ("field_energy", "kinetic_energy", "total_charge"):
            assert abs(dg[k] - do[k]) <= 1e-12 * abs(do[k]), k
